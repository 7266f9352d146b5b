// Adjoint of the estimator for a loss L = sum_b g_b B_b (g = dL/dB):
//   B_b = c_n S_b / (N^3 count_b),  S_b = sum_x prod_t D_{b_t}(x),  c_n = V^{n-1}/N^{3n}
//   G_m(x) = dL/dD_m(x) = sum_b g_b c_n/(N^3 count_b) sum_{t: b_t = m} prod_{u != t} D_{b_u}(x)
//   D_m = inverse(mask_m forward(delta))  =>  dL/d delta(y) = sum_q [mask_{m(q)}(q) Ghat_{m(q)}(q)] e^{+i q.y}
// (the shell kernels are real and even, and the shells are disjoint).
//
// The contraction runs over "entries" e = (m, other factors) with weight
// w_e = sum over the (bin, position) pairs that produce e of g_b / count_b; the
// constant c_n / N^3 is applied when the transformed G_m are gathered.
#include <algorithm>
#include <array>
#include <map>
#include <new>
#include <stdexcept>
#include <vector>

#include "common.cuh"
#include "kernels.h"
#include "plan_internal.h"
#include "tc.cuh"

namespace ps {

constexpr int kAdjWarps = 16;
constexpr int kAdjThreads = 32 * kAdjWarps;
constexpr int kAdjBatch = 8;        // records of one asynchronous copy of weights
constexpr int kAdjRing = 3;         // such batches per warp
constexpr int kAdjMaxTiles = 24;    // tiles of fields in shared memory at most

// A block is 8 consecutive output shells (FP32) or 4 (FP64); a record holds two weights per shell.
// A run of records of one output block: i = i0 .. i0 + count - 1 with the fixed other factors
// (a, j0) and (a, j1) (a: -1 for n = 3; n = 2: no fixed factor at all).
struct AdjSeg {
    short a, j0, j1, i0;
    int count, pad_;
};
struct AdjBlock {  // one output block: its runs, its first record, its record count
    int m0, seg0, nseg, rec0, nrec, pad_[3];
};

// w_e = sum_{k in [off[e], off[e+1])} g[bin[k]] / count[bin[k]], stored at place[e] (place NULL: at e)
template <typename T>
__global__ void adj_weights_kernel(const double* __restrict__ g, const int64_t* __restrict__ counts,
                                   const int* __restrict__ off, const int* __restrict__ bins, int nent,
                                   const int* __restrict__ place, T* __restrict__ w) {
    for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < nent; e += gridDim.x * blockDim.x) {
        double s = 0.0;
        for (int k = off[e]; k < off[e + 1]; k++) {
            const int b = bins[k];
            if (counts[b] > 0) s += g[b] / (double)counts[b];
        }
        w[place ? place[e] : e] = (T)s;
    }
}

// What a lane holds of one field: its cells of a tile (FP32: 8 of 256 cells in eight 32-cell chunks, read in
// 16-byte pieces so that every eight lanes read 128 contiguous bytes; FP64: one of 32).  FP64 runs at 1/64 of
// the FP32 rate, so its blocks of shells are smaller (fewer products outside the entries: 1.19 instead of 1.39
// per entry at 16 shells) and so are its units of work (at 16^3 the larger ones left most of the device idle).
template <typename T>
struct AdjLane;
template <>
struct AdjLane<float> {
    static constexpr int kBlk = 8, kCells = 8, kChunks = 8;
    static PS_DEV uint32_t offset(int lane, int chunk_bytes) { return (uint32_t)((lane >> 3) * chunk_bytes + (lane & 7) * 16); }
    static PS_DEV int cell(int lane, int i) { return 128 * (i >> 2) + 32 * (lane >> 3) + 4 * (lane & 7) + (i & 3); }
    static PS_DEV void load(uint32_t a, int chunk_bytes, float* v) {
#pragma unroll
        for (int h = 0; h < 2; h++)
            asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];"
                         : "=f"(v[4 * h]), "=f"(v[4 * h + 1]), "=f"(v[4 * h + 2]), "=f"(v[4 * h + 3])
                         : "r"(a + (uint32_t)(h * 4 * chunk_bytes)));
    }
    static constexpr int kPerLoad = 4, kPerStore = 4;  // weights of a 16-byte load, cells of a store
    static PS_DEV void load16(uint32_t a, float* v) {
        asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]) : "r"(a));
    }
    static PS_DEV void store(float* g, const float* v) {  // kPerStore consecutive cells
        *reinterpret_cast<float4*>(g) = make_float4(v[0], v[1], v[2], v[3]);
    }
};
template <>
struct AdjLane<double> {
    static constexpr int kBlk = 4, kCells = 1, kChunks = 1;
    static PS_DEV uint32_t offset(int lane, int) { return (uint32_t)(lane * 8); }
    static PS_DEV int cell(int lane, int) { return lane; }
    static PS_DEV void load(uint32_t a, int, double* v) { asm volatile("ld.shared.f64 %0, [%1];" : "=d"(v[0]) : "r"(a)); }
    static constexpr int kPerLoad = 2, kPerStore = 1;
    static PS_DEV void load16(uint32_t a, double* v) {
        asm volatile("ld.shared.v2.f64 {%0, %1}, [%2];" : "=d"(v[0]), "=d"(v[1]) : "r"(a));
    }
    static PS_DEV void store(double* g, const double* v) { *g = *v; }
};

// G[m][x] = sum_{e of m} w_e prod_{f in factors(e)} D[f][x] for the CUDA cores.
//
// A unit of work is (tile of cells, block of output shells): one warp keeps the (shells x cells per lane) sums
// in registers and walks the block's records; a record is a field i next to two fixed products P0, P1 of the
// other factors (n = 3: D_j, D_{j+1}), and adds each shell's two weights times the two products to its sums.  The weights are
// the same for every lane and are read by broadcast from a small ring that the warp fills from L2 by
// asynchronous copies, eight records at a time; weights of absent entries are zero (64 triangle shells: 1.14
// products per entry).
//
// What bounds it: FMA issue (FP32 158 issue slots a record for 128 multiply-adds and 16 products; six 16-byte
// shared loads, 16 wavefronts against 36 cycles of FMAs): 83 % of the issue slots at 128^3 / 40 shells, 1.9 ms
// there against 17.5 ms of one entry at a time (weights and factors from shared memory for two cells a lane,
// 3 flops an entry).
//
// Blocks are persistent.  Their tiles arrive by one bulk copy each (a tile's chunks are contiguous in the
// cell-tiled layout) into a ring; warps take units from a counter, heavy blocks of shells first, and the warp
// that finishes a tile's last unit starts the copy of the tile that takes its place.
template <typename T, int NPRE>
__global__ void __launch_bounds__(kAdjThreads, 1)
    adj_blocks_kernel(const T* __restrict__ D, int nshell, int64_t ncell, int ntile, const AdjBlock* __restrict__ blocks,
                      int nblk, const AdjSeg* __restrict__ segs, const T* __restrict__ w, int nbuf, long long wait_cycles,
                      T* __restrict__ G, int* __restrict__ err) {
    using Ln = AdjLane<T>;
    constexpr int R = Ln::kCells, kBlk = Ln::kBlk, kRec = 2 * kBlk;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    const int row_bytes = 32 * (int)sizeof(T), chunk_bytes = nshell * row_bytes, tile_bytes = Ln::kChunks * chunk_bytes;
    constexpr int kRecBytes = kRec * (int)sizeof(T), kBatchBytes = kAdjBatch * kRecBytes;
    unsigned char* s_ring = smem_raw + (size_t)nbuf * tile_bytes;
    uint64_t* full = reinterpret_cast<uint64_t*>(s_ring + (size_t)kAdjWarps * kAdjRing * kBatchBytes);
    volatile int* s_issued = reinterpret_cast<volatile int*>(full + kAdjMaxTiles);  // tile whose copy was last started
    int* s_done = const_cast<int*>(s_issued) + kAdjMaxTiles;                        // units done of the tile
    int* s_next = s_done + kAdjMaxTiles;
    volatile int* s_abort = s_next + 1;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int ntl = ((int)blockIdx.x < ntile) ? (ntile - 1 - (int)blockIdx.x) / (int)gridDim.x + 1 : 0;  // this block's tiles
    auto copy_tile = [&](int k) {  // one thread
        const int b = k % nbuf;
        tc::mbar_arrive_expect_tx(&full[b], (uint32_t)tile_bytes);
        tc::bulk_load(smem_raw + (size_t)b * tile_bytes,
                      D + ((size_t)blockIdx.x + (size_t)k * gridDim.x) * (tile_bytes / sizeof(T)), (uint32_t)tile_bytes, &full[b]);
        s_issued[b] = k;
    };
    if (threadIdx.x == 0) {
        for (int b = 0; b < nbuf; b++) {
            tc::mbar_init(&full[b], 1);
            s_issued[b] = -1;
            s_done[b] = 0;
        }
        *s_next = 0;
        *s_abort = 0;
        tc::mbar_fence_init();
        for (int k = 0; k < nbuf && k < ntl; k++) copy_tile(k);
    }
    __syncthreads();
    const uint32_t smem = tc::smem_u32(smem_raw);
    const uint32_t ring = tc::smem_u32(s_ring) + (uint32_t)(warp * kAdjRing * kBatchBytes);

    while (true) {
        int u = 0;
        if (lane == 0) u = atomicAdd(s_next, 1);
        u = __shfl_sync(0xffffffffu, u, 0);
        const int k = u / nblk, buf = k % nbuf;
        if (k >= ntl) break;
        const AdjBlock blk = blocks[u - k * nblk];
        // weights of the block's first records, while the tile may still be on its way
        const int nbatch = (blk.nrec + kAdjBatch - 1) / kAdjBatch;
        const char* wsrc = (const char*)(w + (size_t)blk.rec0 * kRec) + lane * 16;
        auto copy_batch = [&](int b) {
            if (b < nbatch) {
#pragma unroll
                for (int i = 0; i < kBatchBytes / 512; i++)
                    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(
                                     ring + (uint32_t)((b % kAdjRing) * kBatchBytes + i * 512 + lane * 16)),
                                 "l"(wsrc + (size_t)b * kBatchBytes + i * 512)
                                 : "memory");
            }
            asm volatile("cp.async.commit_group;" ::: "memory");
        };
        __syncwarp();  // the last unit's weights have been read by every lane
        copy_batch(0);
        copy_batch(1);
        // the tile before in this buffer is done once other warps' last units of it are, a unit's time at most;
        // tile k's copy has been started then, so the barrier's phase before it is over and its parity is unambiguous
        const long long t0 = clock64();
        bool ok = true;
        while (ok && !__all_sync(0xffffffffu, s_issued[buf] == k)) {
            if (*s_abort || clock64() - t0 > wait_cycles) *s_abort = 1;
            ok = !__any_sync(0xffffffffu, *s_abort);
        }
        if (!ok || !tc::mbar_wait_warp(&full[buf], (uint32_t)((k / nbuf) & 1), s_abort)) {
            asm volatile("cp.async.wait_all;" ::: "memory");
            break;
        }
        const uint32_t base = smem + (uint32_t)(buf * tile_bytes) + Ln::offset(lane, chunk_bytes);

        T acc[kBlk][R];
#pragma unroll
        for (int m = 0; m < kBlk; m++)
#pragma unroll
            for (int c = 0; c < R; c++) acc[m][c] = 0;
        int rec = 0;
        uint32_t wp = 0;
        for (int sg = 0; sg < blk.nseg; sg++) {
            const AdjSeg seg = segs[blk.seg0 + sg];
            T P[2][R];
            if constexpr (NPRE >= 1) {
                Ln::load(base + (uint32_t)(seg.j0 * row_bytes), chunk_bytes, P[0]);
                Ln::load(base + (uint32_t)(seg.j1 * row_bytes), chunk_bytes, P[1]);
            }
            if constexpr (NPRE >= 2) {
                T a[R];
                Ln::load(base + (uint32_t)(seg.a * row_bytes), chunk_bytes, a);
#pragma unroll
                for (int c = 0; c < R; c++) {
                    P[0][c] *= a[c];
                    P[1][c] *= a[c];
                }
            }
            uint32_t di = base + (uint32_t)(seg.i0 * row_bytes);
            for (int r = 0; r < seg.count; r++, rec++, di += (uint32_t)row_bytes) {
                if (rec % kAdjBatch == 0) {  // the next batch of weights: landed for every lane; the one after is started
                    const int b = rec / kAdjBatch;
                    asm volatile("cp.async.wait_group 1;" ::: "memory");
                    __syncwarp();
                    copy_batch(b + 2);
                    wp = ring + (uint32_t)((b % kAdjRing) * kBatchBytes);
                }
                T d[R];
                Ln::load(di, chunk_bytes, d);
#pragma unroll
                for (int h = 0; h < (NPRE ? 2 : 1); h++) {
                    T p[R];
#pragma unroll
                    for (int c = 0; c < R; c++) p[c] = NPRE ? P[h][c] * d[c] : d[c];
#pragma unroll
                    for (int m = 0; m < kBlk; m += Ln::kPerLoad) {
                        T wt[Ln::kPerLoad];
                        Ln::load16(wp + (uint32_t)((h * kBlk + m) * sizeof(T)), wt);
#pragma unroll
                        for (int q = 0; q < Ln::kPerLoad; q++)
#pragma unroll
                            for (int c = 0; c < R; c++) acc[m + q][c] = fma(wt[q], p[c], acc[m + q][c]);
                    }
                }
                wp += (uint32_t)kRecBytes;
            }
        }
        const int64_t cell0 = ((int64_t)blockIdx.x + (int64_t)k * gridDim.x) * (Ln::kChunks * 32);
#pragma unroll
        for (int m = 0; m < kBlk; m++)
            if (blk.m0 + m < nshell) {
#pragma unroll
                for (int c = 0; c < R; c += Ln::kPerStore)
                    Ln::store(G + (size_t)(blk.m0 + m) * ncell + cell0 + Ln::cell(lane, c), &acc[m][c]);
            }
        // the tile's reads of this warp are over; its last unit frees the buffer for tile k + nbuf
        __threadfence_block();
        __syncwarp();
        if (lane == 0 && atomicAdd(&s_done[buf], 1) == nblk - 1) {
            s_done[buf] = 0;
            __threadfence_block();
            if (k + nbuf < ntl) copy_tile(k + nbuf);
        }
        __syncwarp();
    }
    __syncthreads();
    if (threadIdx.x == 0 && *s_abort) {
        // every copy started lands before the block exits
        for (int b = 0; b < nbuf; b++)
            if (s_issued[b] >= 0) {
                volatile int no_abort = 0;
                tc::mbar_wait(&full[b], (uint32_t)((s_issued[b] / nbuf) & 1), &no_abort);
            }
        atomicExch(err, tc::kErrTimeout);
    }
}

// H[line][kx] = scale * F[line][kx] for the modes of one shell (its line runs)
template <typename T>
__global__ void shell_gather_kernel(const Cx<T>* __restrict__ F, const short4* __restrict__ lines, int lb, int le,
                                    int K, T scale, Cx<T>* __restrict__ H) {
    const int nk = 2 * K + 1;
    for (int li = lb + blockIdx.x * blockDim.y + threadIdx.y; li < le; li += gridDim.x * blockDim.y) {
        const short4 L = lines[li];
        const size_t base = ((size_t)(L.x + K) * (K + 1) + L.y) * nk + K;
        const int len = L.w - L.z + 1;            // kx in [a, b]
        const int an = L.z > 0 ? L.z : 1;
        const int len2 = L.w >= an ? L.w - an + 1 : 0;  // kx in [-b, -max(a, 1)]
        for (int t = threadIdx.x; t < len + len2; t += blockDim.x) {
            const int kx = t < len ? L.z + t : -(an + (t - len));
            const Cx<T> v = F[base + kx];
            H[base + kx] = cx<T>(v.re * scale, v.im * scale);
        }
    }
}

}  // namespace ps

using namespace ps;

// host -------------------------------------------------------------------------------
struct AtState;  // adjoint_tc.cu
poly_status ps_at_prepare(PsPlan* p, const std::vector<int>& ent_m, const std::vector<short4>& ent, AtState** out);
cudaError_t ps_at_contract(PsPlan* p, AtState* S, const float* w, cudaStream_t st);
int ps_at_error(AtState* S);
void ps_at_free(AtState* S);

struct AdjTables {
    int nent = 0;
    void* d_Wall = nullptr;      // batched forward transforms of the G_m: intermediates and spectra, or NULL
    void* d_fhat_all = nullptr;
    AtState* at = nullptr;  // tensor-core form of the per-cell contraction (bispectrum, split-BF16)
    void *d_eoff = nullptr, *d_ebins = nullptr, *d_w = nullptr;
    // the CUDA-core form: output blocks (heaviest first), their runs of records, every entry's weight's place
    void *d_blocks = nullptr, *d_segs = nullptr, *d_place = nullptr;
    int nblk = 0, nbuf = 1;
    long long wait_cycles = 0;
    size_t nweight = 0, smem = 0;
    int* d_err = nullptr;
    std::vector<int> line_off;  // host copy of the plan's line offsets
};

// The adjoint's entries: one per (m, sorted other shells) that some bin holds,
// grouped by m (moff), each listing its bins once per position of m in the bin
// (eoff / ebins).  Host only.
void ps_adj_entries(const PsPlan* p, std::vector<int>& moff, std::vector<short4>& ent, std::vector<int>& eoff,
                    std::vector<int>& ebins) {
    const int n = p->order;  // 2 .. 4
    // one record per (bin, position t of m in it): key (m, the other shells sorted, -1 padded), bin; sorted
    // stably by key, so each entry's bins keep the (bin, position) order they were produced in
    struct Rec {
        std::array<int, 4> key;
        int bin;
    };
    std::vector<Rec> recs;
    recs.reserve((size_t)p->nbins * n);
    for (int64_t b = 0; b < p->nbins; b++) {
        const int32_t* k = &p->bins[b * n];
        for (int t = 0; t < n; t++) {
            Rec r{{k[t] - 1, -1, -1, -1}, (int)b};
            int c = 1;
            for (int u = 0; u < n; u++)
                if (u != t) r.key[c++] = k[u] - 1;
            std::sort(r.key.begin() + 1, r.key.begin() + n);
            recs.push_back(r);
        }
    }
    std::stable_sort(recs.begin(), recs.end(), [](const Rec& x, const Rec& y) { return x.key < y.key; });
    moff.assign(p->nshell + 1, 0);
    eoff.assign(1, 0);
    ebins.clear();
    ent.clear();
    for (size_t i = 0; i < recs.size();) {  // key order: grouped by m ascending
        const std::array<int, 4>& key = recs[i].key;
        size_t j = i;
        while (j < recs.size() && recs[j].key == key) ebins.push_back(recs[j++].bin);
        moff[key[0] + 1]++;
        short4 f;
        f.x = (short)key[1];
        f.y = (short)key[2];
        f.z = (short)key[3];
        f.w = 0;
        ent.push_back(f);
        eoff.push_back((int)ebins.size());
        i = j;
    }
    for (int m = 0; m < p->nshell; m++) moff[m + 1] += moff[m];
}

// Blocks, runs of records and weight places of the CUDA-core form.  An entry (m, x <= y <= z) is the record
// i = x of the run (block m / blk, a = z, j pair y / 2) (n = 3: no a; n = 2: neither), the weight of m % blk in
// the half y % 2.  A run covers every i from its first to its last; places of absent entries stay zero.  Each
// block's records are padded to whole batches.  Host only.
static void adj_blocks(int order, int nshell, int blk, const std::vector<int>& moff, const std::vector<short4>& ent,
                       std::vector<AdjBlock>& blocks, std::vector<AdjSeg>& segs, std::vector<int>& place, size_t& nweight) {
    struct Rec {
        std::array<int, 3> key;  // block, a, j pair
        int i, j, m, e;
    };
    std::vector<Rec> recs;
    recs.reserve(ent.size());
    for (int m = 0; m < nshell; m++)
        for (int e = moff[m]; e < moff[m + 1]; e++) {
            const int i = ent[e].x, j = order >= 3 ? ent[e].y : 0, a = order == 4 ? ent[e].z : -1;
            recs.push_back({{m / blk, a, j / 2}, i, j, m, e});
        }
    std::stable_sort(recs.begin(), recs.end(), [](const Rec& x, const Rec& y) { return x.key < y.key; });
    place.assign(ent.size(), 0);
    int64_t rec = 0;
    size_t k = 0;
    for (int b = 0; b < (nshell + blk - 1) / blk; b++) {  // every block: one without entries writes zeros
        AdjBlock B{};
        B.m0 = b * blk;
        B.seg0 = (int)segs.size();
        B.rec0 = (int)rec;
        while (k < recs.size() && recs[k].key[0] == b) {
            size_t k1 = k;
            int lo = recs[k].i, hi = recs[k].i;
            for (; k1 < recs.size() && recs[k1].key == recs[k].key; k1++) {
                lo = std::min(lo, recs[k1].i);
                hi = std::max(hi, recs[k1].i);
            }
            AdjSeg S{};
            S.a = (short)recs[k].key[1];
            S.j0 = (short)(2 * recs[k].key[2]);
            S.j1 = (short)std::min(S.j0 + 1, nshell - 1);
            S.i0 = (short)lo;
            S.count = hi - lo + 1;
            for (; k < k1; k++)
                place[recs[k].e] = (int)((rec + recs[k].i - lo) * 2 * blk + recs[k].j % 2 * blk + recs[k].m % blk);
            segs.push_back(S);
            rec += S.count;
            if (rec * 2 * blk > INT32_MAX / 2) throw std::length_error("adjoint: too many weights");
        }
        B.nseg = (int)segs.size() - B.seg0;
        B.nrec = (int)rec - B.rec0;
        rec = (rec + kAdjBatch - 1) / kAdjBatch * kAdjBatch;
        blocks.push_back(B);
    }
    nweight = (size_t)(std::max<int64_t>(kAdjBatch, rec) * 2 * blk);
    std::stable_sort(blocks.begin(), blocks.end(), [](const AdjBlock& x, const AdjBlock& y) { return x.nrec > y.nrec; });
}

// Limit of a warp's wait for a tile buffer: the usual budget and four times the longest unit with every warp at work.
// A record takes 158 issue slots of 16 warps on 4 schedulers in FP32; in FP64 10 instructions of 16 cycles, 16 warps on
// one unit (1/64 of the FP32 rate).  The largest plans of order 4 (128 shells, 179,000 records) hold a unit for 5e8 cycles.
static long long adj_wait_cycles(const std::vector<AdjBlock>& blocks, int is_double) {
    const long long nrec = blocks.empty() ? 0 : blocks[0].nrec;  // heaviest first
    return tc::kWaitBudgetCycles + 4 * nrec * (is_double ? 10 * 16 * 16 : 158 * 16 / 4);
}

extern "C" int poly_diag_adj_blocks(int N, int order, const double* edges, int nshell, unsigned flags, int prec,
                                    int64_t* sizes, int32_t* blocks, int32_t* segs, int32_t* place) {
    if (!sizes) return POLY_ERR_ARG;
    if (order > 4) return POLY_ERR_UNSUPPORTED;  // as poly_backward
    try {
        PsPlan hp;  // host tables only: no device call, no device memory
        std::vector<short> lines;
        if (poly_status s = ps_plan_host_tables(&hp, N, 1.0, order, nshell, edges, (poly_precision)prec, flags, 0, lines))
            return s;
        std::vector<int> mo, eo, eb, at;
        std::vector<short4> en;
        ps_adj_entries(&hp, mo, en, eo, eb);
        std::vector<AdjBlock> B;
        std::vector<AdjSeg> G;
        size_t nweight = 0;
        const int blk = hp.is_double ? AdjLane<double>::kBlk : AdjLane<float>::kBlk;
        adj_blocks(order, nshell, blk, mo, en, B, G, at, nweight);
        const int64_t n[6] = {(int64_t)B.size(), (int64_t)G.size(), (int64_t)at.size(), (int64_t)nweight, blk,
                              adj_wait_cycles(B, hp.is_double)};
        for (int i = 0; i < 6; i++) sizes[i] = n[i];
        for (size_t b = 0; blocks && b < B.size(); b++) {
            const int32_t v[5] = {B[b].m0, B[b].seg0, B[b].nseg, B[b].rec0, B[b].nrec};
            std::copy(v, v + 5, blocks + 5 * b);
        }
        for (size_t g = 0; segs && g < G.size(); g++) {
            const int32_t v[5] = {G[g].a, G[g].j0, G[g].j1, G[g].i0, G[g].count};
            std::copy(v, v + 5, segs + 5 * g);
        }
        if (place) std::copy(at.begin(), at.end(), place);
        return POLY_OK;
    } catch (const std::bad_alloc&) {
        return POLY_ERR_ALLOC;
    } catch (const std::length_error&) {
        return POLY_ERR_UNSUPPORTED;
    }
}

static poly_status adj_prepare(PsPlan* p, AdjTables& A) {
    const int n = p->order;
    std::vector<int> moff, eoff, ebins;
    std::vector<short4> ent;
    ps_adj_entries(p, moff, ent, eoff, ebins);
    A.nent = (int)ent.size();
    if (n == 3 && p->prec == POLY_SPLIT_BF16) {
        std::vector<int> ent_m(ent.size());
        for (int m = 0; m < p->nshell; m++)
            for (int e = moff[m]; e < moff[m + 1]; e++) ent_m[e] = m;
        poly_status s = ps_at_prepare(p, ent_m, ent, &A.at);
        if (s && s != POLY_ERR_UNSUPPORTED) return s;  // unsupported: the CUDA-core kernel below serves
    }
    const size_t es = p->is_double ? 8 : 4;
    auto up = [&](void** d, const void* h, size_t bytes) -> poly_status {
        poly_status s = ps_alloc(p, d, bytes);
        if (s) return s;
        return cudaMemcpy(*d, h, bytes, cudaMemcpyHostToDevice) ? POLY_ERR_CUDA : POLY_OK;
    };
    poly_status s;
    if ((s = up(&A.d_eoff, eoff.data(), eoff.size() * 4)) ||
        (s = up(&A.d_ebins, ebins.data(), std::max<size_t>(1, ebins.size()) * 4)))
        return s;
    A.nweight = std::max(1, A.nent);
    if (!A.at) {
        std::vector<AdjBlock> blocks;
        std::vector<AdjSeg> segs;
        std::vector<int> place;
        const int bs = p->is_double ? AdjLane<double>::kBlk : AdjLane<float>::kBlk;
        adj_blocks(n, p->nshell, bs, moff, ent, blocks, segs, place, A.nweight);
        A.nblk = (int)blocks.size();
        A.wait_cycles = adj_wait_cycles(blocks, p->is_double);
        const size_t tile = (p->is_double ? AdjLane<double>::kChunks : AdjLane<float>::kChunks) * (size_t)p->nshell * 32 * es;
        const size_t rest = (size_t)kAdjWarps * kAdjRing * kAdjBatch * 2 * bs * es + kAdjMaxTiles * 16 + 64;
        A.nbuf = (int)std::max<size_t>(1, std::min<size_t>(kAdjMaxTiles, (224 * 1024 - rest) / tile));
        A.smem = (size_t)A.nbuf * tile + rest;
        if ((s = up(&A.d_blocks, blocks.data(), blocks.size() * sizeof(AdjBlock))) ||
            (s = up(&A.d_segs, segs.data(), std::max<size_t>(1, segs.size()) * sizeof(AdjSeg))) ||
            (s = up(&A.d_place, place.data(), std::max<size_t>(1, place.size()) * 4)) ||
            (s = ps_alloc(p, (void**)&A.d_err, 16)))
            return s;
        if (cudaMemset(A.d_err, 0, 16)) return POLY_ERR_CUDA;
    }
    if ((s = ps_alloc(p, &A.d_w, A.nweight * es))) return s;
    if (cudaMemset(A.d_w, 0, A.nweight * es)) return POLY_ERR_CUDA;  // absent entries stay zero
    A.line_off.resize(p->nshell + 2);
    if (cudaMemcpy(A.line_off.data(), p->d_line_off, (p->nshell + 2) * sizeof(int), cudaMemcpyDeviceToHost))
        return POLY_ERR_CUDA;
    const size_t n3 = (size_t)p->N * p->N * p->N;
    const size_t nl = (size_t)(2 * p->K + 1) * (p->K + 1) * (2 * p->K + 1);
    if ((s = ps_alloc(p, &p->d_G, (size_t)p->nshell * n3 * es))) return s;
    if ((s = ps_alloc(p, &p->d_ghat, nl * 2 * es))) return s;
    // the G_m's forward transforms in one batch when their planes fit shared memory (no spill buffer)
    if (ps_plane_needs_spill(p->N, p->K, p->is_double) == 0) {
        const size_t wsz = (size_t)p->N * (2 * p->K + 1) * (p->K + 1);
        if ((s = ps_alloc(p, &A.d_Wall, (size_t)p->nshell * wsz * 2 * es)) ||
            (s = ps_alloc(p, &A.d_fhat_all, (size_t)p->nshell * nl * 2 * es)))
            return s;
    }
    return POLY_OK;
}

poly_status ps_backward_impl(PsPlan* p, const void* delta, const double* dL_dB, void* dL_ddelta, cudaStream_t st) {
    if (p->order > 4 || p->ell != 0) {
        ps_set_last_error("poly_backward supports monopole plans of orders 2 to 4");
        return POLY_ERR_UNSUPPORTED;
    }
    if (!p->adj) {
        AdjTables* A = new (std::nothrow) AdjTables();
        if (!A) return POLY_ERR_ALLOC;
        poly_status s = adj_prepare(p, *A);
        if (s) {  // the tables' device buffers stay on the plan's list until it is destroyed
            ps_at_free(A->at);
            delete A;
            return s;
        }
        p->adj = A;
    }
    AdjTables& A = *p->adj;
    poly_status s = ps_fields(p, delta, st);
    if (s) return s;
    const int64_t ncell = (int64_t)p->N * p->N * p->N;
    const int dbl = p->is_double;
    cudaError_t e;
    const int wb = std::max(1, std::min(4096, (A.nent + 255) / 256));
    if (dbl)
        adj_weights_kernel<double><<<wb, 256, 0, st>>>(dL_dB, p->d_counts, (const int*)A.d_eoff, (const int*)A.d_ebins,
                                                       A.nent, (const int*)A.d_place, (double*)A.d_w);
    else
        adj_weights_kernel<float><<<wb, 256, 0, st>>>(dL_dB, p->d_counts, (const int*)A.d_eoff, (const int*)A.d_ebins,
                                                      A.nent, (const int*)A.d_place, (float*)A.d_w);
    if (A.at) {
        if ((e = ps_at_contract(p, A.at, (const float*)A.d_w, st))) return POLY_ERR_CUDA;
    } else {
        auto go = [&](auto kern, auto zero) -> cudaError_t {
            using T = decltype(zero);
            cudaError_t e2 = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)A.smem);
            if (e2) return e2;
            const int ntile = (int)(ncell / (AdjLane<T>::kChunks * 32));  // N^3 is a multiple of 256
            kern<<<std::min(p->sms, ntile), kAdjThreads, A.smem, st>>>(
                (const T*)p->d_fields, p->nshell, ncell, ntile, (const AdjBlock*)A.d_blocks, A.nblk, (const AdjSeg*)A.d_segs,
                (const T*)A.d_w, A.nbuf, A.wait_cycles, (T*)p->d_G, A.d_err);
            return cudaSuccess;
        };
        if (dbl)
            e = p->order == 2 ? go(adj_blocks_kernel<double, 0>, 0.0)
                              : p->order == 3 ? go(adj_blocks_kernel<double, 1>, 0.0) : go(adj_blocks_kernel<double, 2>, 0.0);
        else
            e = p->order == 2 ? go(adj_blocks_kernel<float, 0>, 0.f)
                              : p->order == 3 ? go(adj_blocks_kernel<float, 1>, 0.f) : go(adj_blocks_kernel<float, 2>, 0.f);
        if (e) return POLY_ERR_CUDA;
    }
    if ((e = cudaGetLastError())) return POLY_ERR_CUDA;
    p->launches += A.at ? 3 : 2;
    // H = c_n / N^3 * sum_m mask_m forward(G_m)
    const size_t nl = (size_t)(2 * p->K + 1) * (p->K + 1) * (2 * p->K + 1);
    const size_t es = dbl ? 8 : 4;
    if ((e = cudaMemsetAsync(p->d_ghat, 0, nl * 2 * es, st))) return POLY_ERR_CUDA;
    const double scale = ps_norm(p) / (double)ncell;
    // forward transforms of all G_m: one batched launch pair when the per-field outputs fit (A.d_Wall), else
    // one field at a time through the plan's workspace
    const bool batched = A.d_Wall != nullptr;
    if (batched) {
        if ((e = ps_forward_batched(p->N, dbl, p->d_G, p->nshell, p->K, p->d_tw_fwd, A.d_Wall, A.d_fhat_all, nullptr,
                                    st)))
            return POLY_ERR_CUDA;
        p->launches += 2;
    }
    for (int m = 0; m < p->nshell; m++) {
        const void* Gm = (const char*)p->d_G + (size_t)m * ncell * es;
        const void* Fm = batched ? (const void*)((const char*)A.d_fhat_all + (size_t)m * nl * 2 * es) : p->d_fhat;
        if (!batched) {
            if ((e = ps_forward(p->N, dbl, Gm, p->K, p->d_tw_fwd, p->d_W, p->d_fhat, p->d_spill, st)))
                return POLY_ERR_CUDA;
            p->launches += 2;
        }
        const int lb = A.line_off[m], le = A.line_off[m + 1];
        if (le > lb) {
            dim3 blk(32, 8);
            const unsigned nb = (unsigned)std::min(1024, (le - lb + 7) / 8);
            if (dbl)
                shell_gather_kernel<double><<<nb, blk, 0, st>>>((const Cx<double>*)Fm, (const short4*)p->d_lines,
                                                               lb, le, p->K, scale, (Cx<double>*)p->d_ghat);
            else
                shell_gather_kernel<float><<<nb, blk, 0, st>>>((const Cx<float>*)Fm, (const short4*)p->d_lines,
                                                              lb, le, p->K, (float)scale, (Cx<float>*)p->d_ghat);
            if ((e = cudaGetLastError())) return POLY_ERR_CUDA;
        }
        p->launches += 1;
    }
    // one inverse transform over the union of the shells
    if (!ps_xpre_fits(p, p->nshell, 1)) return POLY_ERR_ARG;
    if ((e = ps_inverse(p->N, dbl, 0, p->d_ghat, p->d_lines, p->d_line_off, p->nshell, 1, p->K, 0, p->N, p->d_tw_inv,
                        dL_ddelta, (size_t)ncell, p->d_spill, p->d_xpre, p->max_lines, 0, st)))
        return POLY_ERR_CUDA;
    p->launches += 2;
    return POLY_OK;
}

void ps_adj_free(PsPlan* p) {
    if (p->adj) ps_at_free(p->adj->at);
    delete p->adj;
    p->adj = nullptr;
}

int ps_adj_device_error(PsPlan* p) {
    if (!p->adj) return 0;
    if (p->adj->at) return ps_at_error(p->adj->at);
    int v = 0;
    if (!p->adj->d_err || cudaMemcpy(&v, p->adj->d_err, 4, cudaMemcpyDeviceToHost)) return 0;
    if (v) cudaMemset(p->adj->d_err, 0, 4);
    return v;
}
