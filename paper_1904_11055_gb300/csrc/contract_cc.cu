// CUDA-core contraction over grid cells (Eq. estimator, discrete form of App. A):
//   S_b = sum_x prod_t D_{b_t}(x)
//
// A task is a block of bins: one run of consecutive shells per leg (e.g. 4 x 4 x 4
// for FP32 bispectra), rows the products of the first legs and columns the
// products of the rest.  One warp takes a task and its lanes the cells: each lane
// loads one value (FP32: of two neighbouring cells) per field of the task's runs,
// forms the row and column products in registers and adds every row times every
// column to its own accumulators, kept in registers over all of the warp's cells.
// FP32 arithmetic runs in packed pairs, one cell in each half, so that no operand
// has to be duplicated.
//
// What bounds it: latency, of the factors' shared-memory loads and of the row and column products in front of the
// multiply-adds, at the 12 warps an SM that 168 registers a thread leave: at 160^3 / 48 shells 48 % of the issue slots
// and a third of the FMA pipe are busy.  The shared memory is not the bound: the block over three legs needs 24
// wavefronts (4 + 4 + 4 fields, conflict-free rows of the cell-tiled layout) for
// 64 + 16 packed multiply-adds and products, 60 % of its rate at
// the FP32 FMA peak.  (A 64 x 64 tile of products staged in shared memory, 4 x 4
// per lane and two 16-byte loads per 16 FMAs, is bound by those loads at 50 % of the
// peak before the products and the idle parts of the tile: 121 ms at 256^3 / 64
// shells against 35.5 ms here, 38 TFLOP/s (31 without the products) of a measured 56 to 66 TFLOP/s of packed
// FMAs over such register blocks; FP64 at 64^3 / 16 shells 1.05 against 0.45 ms.)
// The blocks follow the bins closely: 508 tasks x 64 = 1.33 products per bin at
// 24,432 triangles.
//
// Fields of one block's tasks arrive by 16-byte asynchronous copies of every thread
// (stages of a few chunks) and serve its 12 warps; one bulk copy per run of fields
// and chunk, about a KB each, took 58 ms.  FP32 lane sums cover 256 steps (two
// sums, of the even and the odd cells); then they are added over the warp with their rounding errors and go to FP64
// sums.  FP64 throughout for the plain
// method and the exact polygon counts over the symmetry wedge (cell weights on the
// rows).
#include <algorithm>
#include <type_traits>

#include "common.cuh"
#include "kernels.h"

namespace ps {

constexpr int kCcWarps = kCcTasksPerGroup;                          // task warps per block
constexpr int kCcThreads = kCcWarps * 32;
constexpr int kCcFlush = 256;  // steps per FP32 partial sum

PS_DEV void cc_copy16(uint32_t dst_smem, const void* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst_smem), "l"(src) : "memory");
}
PS_DEV void cc_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int LEFT>
PS_DEV void cc_wait() {  // all but this thread's last LEFT groups of copies have landed
    asm volatile("cp.async.wait_group %0;" ::"n"(LEFT) : "memory");
}

// What a lane holds of one field in one step: two cells (FP32) or one (FP64).
template <typename T>
struct CcLane;
template <>
struct CcLane<float> {
    using V = unsigned long long;  // two floats; as one 64-bit value they stay in an aligned register pair without moves
    static constexpr int kChunks = 2;  // 32-cell chunks of a step: lanes 0-15 take the first, 16-31 the second
    static PS_DEV uint32_t offset(int lane, int chunk_bytes) { return (uint32_t)((lane >> 4) * chunk_bytes + (lane & 15) * 8); }
    static PS_DEV V zero() { return 0ull; }
    static PS_DEV V load(uint32_t a) {
        V v;
        asm volatile("ld.shared.b64 %0, [%1];" : "=l"(v) : "r"(a));
        return v;
    }
    static PS_DEV V mul(V a, V b) {
        V r;
        asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
        return r;
    }
    static PS_DEV V mad(V a, V b, V c) {
        asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(c) : "l"(a), "l"(b));
        return c;
    }
    static PS_DEV V abs(V a) { return a & 0x7fffffff7fffffffull; }
    static PS_DEV float lo(V a) { return __uint_as_float((uint32_t)a); }
    static PS_DEV float hi(V a) { return __uint_as_float((uint32_t)(a >> 32)); }
};
template <>
struct CcLane<double> {
    using V = double;
    static constexpr int kChunks = 1;
    static PS_DEV uint32_t offset(int lane, int) { return (uint32_t)(lane * 8); }
    static PS_DEV V zero() { return 0.0; }
    static PS_DEV V load(uint32_t a) {
        V v;
        asm volatile("ld.shared.f64 %0, [%1];" : "=d"(v) : "r"(a));
        return v;
    }
    static PS_DEV V mul(V a, V b) { return a * b; }
    static PS_DEV V mad(V a, V b, V c) { return fma(a, b, c); }
    static PS_DEV V abs(V a) { return fabs(a); }
};

// The products of one value per leg of legs [L0, L1), the first leg's index slowest; leg l's values at d[S::at(l)].
template <typename T, class S, int L0, int L1>
PS_DEV void cc_products(const typename CcLane<T>::V* d, typename CcLane<T>::V* o) {
    constexpr int D = S::dim(L1 - 1), n = S::span(L0, L1 - 1), at = S::at(L1 - 1);
    if constexpr (L1 - L0 == 1) {
#pragma unroll
        for (int i = 0; i < D; i++) o[i] = d[at + i];
    } else {
        typename CcLane<T>::V h[n];
        cc_products<T, S, L0, L1 - 1>(d, h);
#pragma unroll
        for (int a = 0; a < n; a++)
#pragma unroll
            for (int i = 0; i < D; i++) o[a * D + i] = CcLane<T>::mul(h[a], d[at + i]);
    }
}

// a + b: the rounded sum, and in e its rounding error (Knuth's two-sum; not a number where the sum is infinite).
PS_DEV float cc_two_sum(float a, float b, float& e) {
    const float s = __fadd_rn(a, b), t = __fsub_rn(s, a);
    e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, t)), __fsub_rn(b, t));
    return s;
}

// Sum of V values over the warp's 32 lanes by halving: after the exchange at lane distance d a
// lane keeps the half of the values that its bit d selects.  V = 64: lane l ends with values
// 2 l' and 2 l' + 1, l' = the bits of l (16 first) as the high bits of the value index.  FP32
// values carry their sum's rounding error beside them (e), so that what FP64 takes over is the
// lanes' sums added to about 48 bits; adding them in FP64 costs 8 % (256^3 / 64 shells 37.3 and 40.7 ms).
template <typename T, int V>
PS_DEV void cc_warp_sum(T* v, T* e, int lane) {
    int n = V;
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) {
        const bool halve = n > 1, up = halve && (lane & d);
        if (halve) n >>= 1;
#pragma unroll
        for (int i = 0; i < V / 2; i++)
            if (i < n) {
                const int k = halve ? i + n : i;
                const T keep = up ? v[k] : v[i], give = up ? v[i] : v[k];
                const T other = __shfl_xor_sync(0xffffffffu, give, d);
                if constexpr (sizeof(T) == 4) {
                    const T ekeep = up ? e[k] : e[i], egive = up ? e[i] : e[k];
                    T err;
                    v[i] = cc_two_sum(keep, other, err);
                    e[i] = ekeep + __shfl_xor_sync(0xffffffffu, egive, d) + err;
                } else {
                    v[i] = keep + other;
                }
            }
    }
}

template <typename T, int ORDER, bool WEIGHTED, bool ABS>
__global__ void __launch_bounds__(kCcThreads, 1)
    contract_cc_kernel(const T* __restrict__ fields, int nf, int64_t nchunk, const T* __restrict__ weight,
                       const CcGroup* __restrict__ groups, int ngroups, const CcTask* __restrict__ tasks, int64_t ntask,
                       int nsplit, int wpt, int stage_chunks, int stage_bytes, double* __restrict__ partial) {
    using S = CcShape<ORDER, sizeof(T) == 8>;
    using Ln = CcLane<T>;
    using LV = typename Ln::V;
    constexpr int RA = S::ra, V = S::rows * S::cols;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int gi = blockIdx.x % ngroups, split = blockIdx.x / ngroups;
    const CcGroup* grp = groups + gi;
    const int used = grp->used, task_off = grp->task_off, tpg = grp->ntask;
    // the block's chunks (whole steps), in stages
    const int64_t nstep = nchunk / Ln::kChunks;
    const int64_t c0 = nstep * split / nsplit * Ln::kChunks, c1 = nstep * (split + 1) / nsplit * Ln::kChunks;
    const int nst = (int)((c1 - c0 + stage_chunks - 1) / stage_chunks);
    const int row_bytes = 32 * (int)sizeof(T);
    const int chunk_bytes = used * row_bytes;

    // copies of stage `it`: eight threads per field row, 32 rows at a time, chunk by chunk
    const uint32_t smem = (uint32_t)__cvta_generic_to_shared(smem_raw);
    constexpr int kPieces = 32 * sizeof(T) / 16 / 8;  // 16-byte pieces of a row per thread
    auto copy_stage = [&](int it) {
        const int64_t c = c0 + (int64_t)it * stage_chunks;
        const int cnt = (int)(c1 - c < stage_chunks ? c1 - c : stage_chunks);
        for (int u = threadIdx.x >> 3; u < used; u += kCcThreads / 8) {
            uint32_t dst = smem + (uint32_t)((it % kCcStages) * stage_bytes + u * row_bytes + (threadIdx.x & 7) * 16);
            const char* src = (const char*)(fields + ((size_t)c * nf + grp->slot[u]) * 32) + (threadIdx.x & 7) * 16;
            for (int k = 0; k < cnt; k++) {
#pragma unroll
                for (int i = 0; i < kPieces; i++) cc_copy16(dst + i * 128, src + i * 128);
                dst += chunk_bytes;
                src += (size_t)nf * row_bytes;
            }
        }
    };
    for (int it = 0; it < kCcStages - 1; it++) {
        if (it < nst) copy_stage(it);
        cc_commit();
    }
    // ---------------------------------------------------------------- tasks
    const int ti = warp % tpg, phase = warp / tpg;  // warps beyond tpg * wpt only copy
    const bool active = phase < wpt;
    CcTask task;
#pragma unroll
    for (int l = 0; l < ORDER; l++) {
        task.row[l] = tasks[task_off + ti].row[l] * (int)sizeof(T);
    }
    LV acc[S::rows][S::cols];
    double acc64[(V + 31) / 32];
#pragma unroll
    for (int i = 0; i < S::rows; i++)
#pragma unroll
        for (int j = 0; j < S::cols; j++) acc[i][j] = Ln::zero();
#pragma unroll
    for (int i = 0; i < (V + 31) / 32; i++) acc64[i] = 0.0;

    auto flush = [&]() {
        constexpr int E = sizeof(T) == 4 ? V : 1;
        T v[V], e[E];
#pragma unroll
        for (int i = 0; i < S::rows; i++)
#pragma unroll
            for (int j = 0; j < S::cols; j++) {
                const int k = i * S::cols + j;
                if constexpr (sizeof(T) == 4) v[k] = cc_two_sum(Ln::lo(acc[i][j]), Ln::hi(acc[i][j]), e[k]);
                else v[k] = acc[i][j];
                acc[i][j] = Ln::zero();
            }
        cc_warp_sum<T, V>(v, e, lane);
#pragma unroll
        for (int i = 0; i < (V + 31) / 32; i++) {
            acc64[i] += (double)v[i];
            if constexpr (sizeof(T) == 4) acc64[i] += e[i] == e[i] ? (double)e[i] : 0.0;  // an infinite sum has no error term
        }
    };

    const uint32_t p0 = smem + Ln::offset(lane, chunk_bytes);
    const int step_bytes = Ln::kChunks * chunk_bytes;
    int next = phase, since = 0;  // this warp's next step (of the block's range), at least the steps since the last flush
    for (int it = 0; it < nst; it++) {
        cc_wait<kCcStages - 2>();  // stage it has landed
        __syncthreads();           // for every thread, and stage it - 1 has been read by every warp
        if (it + kCcStages - 1 < nst) copy_stage(it + kCcStages - 1);
        cc_commit();
        const int s = it % kCcStages;
        const int spst = stage_chunks / Ln::kChunks, b0 = it * spst;  // steps of a stage, its first step
        const int left = (int)((c1 - c0) / Ln::kChunks) - b0, cnt = left < spst ? left : spst;
        if (active) {
            int k = next - b0;
            uint32_t p = p0 + (uint32_t)(s * stage_bytes + k * step_bytes);
            for (; k < cnt; k += wpt, p += (uint32_t)(wpt * step_bytes)) {
                LV d[S::nval], rows[S::rows], col[S::cols];
#pragma unroll
                for (int l = 0; l < ORDER; l++)
#pragma unroll
                    for (int i = 0; i < S::dim(l); i++)
                        d[S::at(l) + i] = Ln::load(p + task.row[l] + 32 * i * (uint32_t)sizeof(T));
                cc_products<T, S, 0, RA>(d, rows);
                cc_products<T, S, RA, ORDER>(d, col);
                if constexpr (WEIGHTED) {
                    const T w = weight[(c0 + b0 + k) * 32 + lane];
#pragma unroll
                    for (int i = 0; i < S::rows; i++) rows[i] = Ln::mul(rows[i], w);
                }
                if constexpr (ABS) {
#pragma unroll
                    for (int i = 0; i < S::rows; i++) rows[i] = Ln::abs(rows[i]);
#pragma unroll
                    for (int j = 0; j < S::cols; j++) col[j] = Ln::abs(col[j]);
                }
#pragma unroll
                for (int i = 0; i < S::rows; i++)
#pragma unroll
                    for (int j = 0; j < S::cols; j++) acc[i][j] = Ln::mad(rows[i], col[j], acc[i][j]);
            }
            since += cnt;
            next = b0 + k;
        }
        if (sizeof(T) == 4 && since >= kCcFlush) {
            flush();
            since = 0;
        }
    }
    if (active) {
        flush();
        // lane -> value index of cc_warp_sum (the lane's bits, highest first)
        double* out = partial + ((size_t)(split * wpt + phase) * ntask + task_off + ti) * V;
        if constexpr (V >= 32) {
#pragma unroll
            for (int i = 0; i < V / 32; i++) out[lane * (V / 32) + i] = acc64[i];
        } else {
            constexpr int REP = 32 / V;  // lanes that differ in the low bits hold the same value
            if (lane % REP == 0) out[lane / REP] = acc64[0];
        }
    }
}

// out[b] = norm * S_b / (n3 count_b) (0 where the count is 0; counts NULL: S_b), S_b = the sum of partial[k][slot_b]
// over the nsplit rows.  One warp per bin: a bin's rows lie far apart, so what bounds it is the latency of a
// lane's few loads (one thread per bin took 60 us of 300 rows at 3,384 bins).
__global__ void reduce_slots_kernel(const double* __restrict__ partial, int nsplit, int64_t slot_stride,
                                    const int64_t* __restrict__ slot, const int64_t* __restrict__ counts, int64_t nbins,
                                    double norm, double n3, double* __restrict__ out) {
    const int lane = threadIdx.x & 31;
    const int64_t nw = (int64_t)gridDim.x * (blockDim.x >> 5);
    for (int64_t b = blockIdx.x * (int64_t)(blockDim.x >> 5) + (threadIdx.x >> 5); b < nbins; b += nw) {
        const int64_t o = slot[b];
        double s = 0.0;
        for (int k = lane; k < nsplit; k += 32) s += partial[(size_t)k * slot_stride + o];
        s = warp_sum(s);
        if (lane == 0) {
            const int64_t c = counts ? counts[b] : 0;
            out[b] = !counts ? s : c > 0 ? norm * s / (n3 * (double)c) : 0.0;
        }
    }
}

template <typename T, int ORDER>
static cudaError_t contract_cc_launch(const CcLaunch& L, int weighted, int absval, const void* fields, const void* weight,
                                      const CcGroup* groups, const CcTask* tasks, double* partial,
                                      cudaStream_t st) {
    auto go = [&](auto k) -> cudaError_t {
        cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)L.smem_bytes);
        if (e) return e;
        k<<<(unsigned)(L.ngroups * L.nsplit), kCcThreads, L.smem_bytes, st>>>(
            (const T*)fields, L.nf, L.nchunk, (const T*)weight, groups, L.ngroups, tasks, L.ntask, L.nsplit, L.wpt,
            L.stage_chunks, L.stage_bytes, partial);
        return cudaGetLastError();
    };
    if (weighted) {
        if constexpr (sizeof(T) == 8) return go(contract_cc_kernel<T, ORDER, true, false>);
        return cudaErrorInvalidValue;
    }
    return absval ? go(contract_cc_kernel<T, ORDER, false, true>) : go(contract_cc_kernel<T, ORDER, false, false>);
}

}  // namespace ps

using namespace ps;

cudaError_t ps_contract_cc(int is_double, int order, int weighted, int absval, const CcLaunch& L, const void* fields,
                           const void* weight, const CcGroup* groups, const CcTask* tasks, double* partial,
                           cudaStream_t st) {
#define PS_CC(O)                                                                                                       \
    case O:                                                                                                            \
        return is_double ? contract_cc_launch<double, O>(L, weighted, absval, fields, weight, groups, tasks, partial, st) \
                         : contract_cc_launch<float, O>(L, weighted, absval, fields, weight, groups, tasks, partial, st);
    switch (order) { PS_CC(2) PS_CC(3) PS_CC(4) PS_CC(5) PS_CC(6) }
#undef PS_CC
    return cudaErrorInvalidValue;
}

cudaError_t ps_reduce_slots(const double* partial, int nsplit, int64_t slot_stride, const int64_t* slot,
                            const int64_t* counts, int64_t nbins, double norm, double n3, double* out, cudaStream_t st) {
    if (nbins <= 0) return cudaSuccess;
    const int blocks = (int)std::min<int64_t>((nbins + 7) / 8, 8192);
    reduce_slots_kernel<<<blocks, 256, 0, st>>>(partial, nsplit, slot_stride, slot, counts, nbins, norm, n3, out);
    return cudaGetLastError();
}
