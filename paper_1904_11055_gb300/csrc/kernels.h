// Internal launch interface between the plan code and the CUDA kernels.
#pragma once
#include <cuda_runtime.h>
#include <stddef.h>
#include <stdint.h>

// ---- fields.cu --------------------------------------------------------------
int ps_supported_n(int n);
int ps_plane_needs_spill(int n, int K, int is_double);
size_t ps_spill_elems(int n, int K, int nblocks, int is_double);
// delta [N^3] real -> W [N][(2K+1)(K+1)] -> fhat [(2K+1)(K+1)][2K+1] (complex, same precision)
cudaError_t ps_forward(int n, int is_double, const void* delta, int K, const void* tw_fwd, void* W, void* fhat,
                       void* spill, cudaStream_t st);
// the same for nfields fields N^3 apart in one launch pair: W and fhat hold one output per field, N (2K+1)(K+1)
// and (2K+1)(K+1)(2K+1) complex values apart; spill (when needed) nfields * N blocks
cudaError_t ps_forward_batched(int n, int is_double, const void* delta, int nfields, int K, const void* tw_fwd, void* W,
                               void* fhat, void* spill, cudaStream_t st);
// shells s0..s0+ns-1, planes x0..x0+nx-1 -> out[(s-s0)*out_stride + (x-x0)*N*N + y*N + z].
// xpre != NULL (and not unity): first run the x pass into xpre (sum over shells of lines * N complex values;
// max_lines = the largest line count of the shells), then scatter; otherwise gather along x in the plane kernel.
// tile_ns > 0: write the cell-tiled layout out[(cell/32) * tile_ns * 32 + s * 32 + cell % 32] (absolute shell s,
// x0 must be 0) instead of the natural one.
cudaError_t ps_inverse(int n, int is_double, int unity, const void* fhat, const void* lines, const int* line_off,
                       int s0, int ns, int K, int x0, int nx, const void* tw_inv, void* out, size_t out_stride,
                       void* spill, void* xpre, int max_lines, int tile_ns, cudaStream_t st);
// The FP32 estimate-path inverse in runs of shells sized by each shell's largest
// kz (kz_host: host array indexed by shell; kz_dev: the same on the device, or
// NULL); see inverse_ranged_n.
cudaError_t ps_inverse_ranged_f32(int n, const void* fhat, const void* lines, const int* line_off, int s0, int ns, int K,
                                  const void* tw_inv, void* out, size_t out_stride, void* spill, void* xpre,
                                  int max_lines, int tile_ns, const int* kz_host, const int* kz_dev, cudaStream_t st);

// ---- contract_cc.cu -----------------------------------------------------------
// CUDA-core contraction: a task is a block of bins, one run of consecutive field
// slots per leg; row (r) = the products of the first ra legs' runs, column (c) = of
// the rest, the first leg's index slowest, product r * cols + c.  The run lengths per
// order (a nibble per leg, first leg lowest): 64 products for FP32, where longer runs
// save products and loads; 16 for FP64, whose 1/64-rate multiply-adds make every
// product outside the bins dear (64 triangle shells: 1.33 products per bin in FP32,
// 1.16 in FP64; 16 shells: 2.14 and 1.57).
__host__ __device__ constexpr unsigned cc_code(int order, bool dbl) {
    return dbl ? (order == 2 ? 0x44u : order == 3 ? 0x422u : order == 4 ? 0x2222u : order == 5 ? 0x22122u : 0x221221u)
               : (order == 2 ? 0x88u : order == 3 ? 0x444u : order == 4 ? 0x4224u : order == 5 ? 0x42222u : 0x222222u);
}
__host__ __device__ constexpr int cc_ra(int order) { return order <= 2 ? 1 : (order <= 5 ? 2 : 3); }
__host__ __device__ constexpr int cc_dim(int order, bool dbl, int leg) { return (int)((cc_code(order, dbl) >> (4 * leg)) & 15u); }
__host__ __device__ constexpr int cc_span(int order, bool dbl, int l0, int l1) {  // product of the run lengths of legs [l0, l1)
    int n = 1;
    for (int l = l0; l < l1; l++) n *= cc_dim(order, dbl, l);
    return n;
}
__host__ __device__ constexpr int cc_at(int order, bool dbl, int leg) {  // run lengths of the legs before it
    int n = 0;
    for (int l = 0; l < leg; l++) n += cc_dim(order, dbl, l);
    return n;
}
template <int ORDER, bool DBL>
struct CcShape {
    static constexpr int nval = cc_at(ORDER, DBL, ORDER);  // values of a task per cell
    static constexpr int ra = cc_ra(ORDER), rows = cc_span(ORDER, DBL, 0, ra), cols = cc_span(ORDER, DBL, ra, ORDER);
    __host__ __device__ static constexpr int dim(int l) { return cc_dim(ORDER, DBL, l); }
    __host__ __device__ static constexpr int at(int l) { return cc_at(ORDER, DBL, l); }
    __host__ __device__ static constexpr int span(int l0, int l1) { return cc_span(ORDER, DBL, l0, l1); }
};
constexpr int kCcTasksPerGroup = 12;  // the warps of a block: FP32 tasks keep 168 registers a thread (8 warps at 216: 36.0 against 35.8 ms, FP64 0.51 against 0.45 ms)
constexpr int kCcStages = 4;
constexpr int kCcMaxSlots = 192;  // field slots the tasks of a group may name: at most 12 tasks x 16 (two runs of eight)
constexpr int kCcPadRows = 8;   // rows after the last stage that a run past the last field may read (its products are unused)
struct CcTask {
    int row[6];  // per leg: element offset (32 per field row) of its run in the block's copy of a chunk
};
struct CcGroup {  // the tasks of one block
    int task_off, ntask, used;  // used: field rows copied per chunk
    int slot[kCcMaxSlots];      // their field slots, ascending
};
struct CcLaunch {
    int nf = 0;           // field slots of a chunk in the cell-tiled array
    int64_t nchunk = 0;   // 32-cell chunks
    int ngroups = 0;
    int64_t ntask = 0;
    int nsplit = 1, wpt = 1;  // ranges of chunks; warps that share a task
    int stage_chunks = 1, stage_bytes = 0;
    size_t smem_bytes = 0;
    int values = 64;      // products of a task
    int64_t rows() const { return (int64_t)nsplit * wpt; }          // partial sums per task
    int64_t stride() const { return ntask * (int64_t)values; }      // doubles between them
};
// partial[(split * wpt + phase) * stride + task * values + product]: FP64 sums over that part of the cells.
// fields: cell-tiled, [nchunk][nf][32]; weight (FP64 only): [nchunk * 32] cell weights.
cudaError_t ps_contract_cc(int is_double, int order, int weighted, int absval, const CcLaunch& L, const void* fields,
                           const void* weight, const CcGroup* groups, const CcTask* tasks, double* partial,
                           cudaStream_t st);
// out[b] = norm * S_b / (n3 count[b]) (0 where count == 0; counts NULL: S_b), S_b = sum_split partial[split * slot_stride + slot[b]]
cudaError_t ps_reduce_slots(const double* partial, int nsplit, int64_t slot_stride, const int64_t* slot,
                            const int64_t* counts, int64_t nbins, double norm, double n3, double* out, cudaStream_t st);
// disconnected part of the trispectrum: shell powers P (device, nshell) from the pruned spectrum, then B_disc per bin
cudaError_t ps_disconnected(int is_double, const void* fhat, const void* lines, const int* line_off, int nshell, int K,
                            const int32_t* bins, const int64_t* counts, int64_t nbins, double norm, double n3,
                            double* P, double* out, cudaStream_t st);
// out = L_ell(kz/|q|) * fhat over the pruned half spectrum (even ell; the mode q = 0 gets weight 0)
cudaError_t ps_legendre_weight(int is_double, const void* fhat, int K, int ell, void* out, cudaStream_t st);

// ---- misc.cu -------------------------------------------------------------------
// ---- counts_exact.cu ---------------------------------------------------------
// out = F[s0] F[s1] F[s2] (slots -1: none), FP64 fields of n3 cells in natural layout
cudaError_t ps_prod_fields(const double* F, size_t n3, int s0, int s1, int s2, double* out, cudaStream_t st);
// G[i] = round(Re fhat[i] * inv_n3) for n complex FP64 values; *err = 1 if any is not near an integer
cudaError_t ps_round_map(const void* fhat, size_t n, double inv_n3, long long* G, int* err, cudaStream_t st);
// out[b] = sum over the half cube |p_c| <= Kp of w(kz) maps[which[b].x][i] maps[which[b].y][i]
cudaError_t ps_dot_maps(const long long* maps, size_t mapsz, const int2* which, int nbins, int Kp,
                        unsigned long long* out, cudaStream_t st);

// cells idx[w] of ns natural-layout FP64 fields, in_stride apart, into slots s0 .. s0 + ns - 1 of the cell-tiled
// array out[(w / 32) * nf * 32 + slot * 32 + w % 32]; w in [nw, nw rounded up to 32) is set to 0
cudaError_t ps_gather_cells(const double* in, size_t in_stride, int s0, int ns, int nf, const int32_t* idx, int64_t nw,
                            double* out, cudaStream_t st);
