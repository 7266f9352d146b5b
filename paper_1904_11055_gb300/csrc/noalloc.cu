// Bispectrum of a small field without allocating device memory.
//
// Some callers cannot call cudaMalloc when they need an estimate: code that
// runs after a memory budget has been fixed and must not allocate any more, or
// code inside a framework whose device allocator belongs to someone else.
// poly_estimate_noalloc serves them: it runs the same kernels as poly_estimate,
// with every intermediate (twiddles, shell tables, spectrum, shell fields,
// contraction partials, sums, counts) placed in one static device array that
// belongs to this library.
//
// Each call builds its host tables (twiddles, shell line tables, contraction
// tasks) in ordinary pageable host memory and copies them, and the counts, into
// the array with cudaMemcpyAsync.  Copies from pageable memory are staged
// through the driver, so a call can wait for its stream before it returns; it
// is not a zero-latency call.
//
// The array costs kNoAllocBytes on every GPU that loads the library, until the
// process exits.  Its device address is looked up once per device, on the first
// call made with that device current (so make that first call before any stream
// capture).  All calls share the array: two calls whose work overlaps on the
// GPU (different streams, or different host threads) race on it.  Each call
// overwrites every region it reads before reading it, so nothing depends on
// what an earlier call left behind.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <mutex>
#include <new>
#include <stdexcept>
#include <string>
#include <vector>

#include "../../include/polyspec.h"
#include "kernels.h"
#include "plan_internal.h"

namespace {
constexpr size_t kNoAllocBytes = (size_t)32 << 20;  // 32 MiB
constexpr int kMaxDevices = 64;

std::mutex g_setup_mu;
void* g_scratch_addr[kMaxDevices] = {};

poly_status fail(poly_status s, const std::string& msg) {
    ps_set_last_error(msg);  // reported by poly_last_error()
    return s;
}
}  // namespace

static __device__ __align__(256) unsigned char g_noalloc_scratch[kNoAllocBytes];

// Device address of the static array for the current device (looked up once per device).
static poly_status scratch_for_current_device(void** out) {
    int dev = -1;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return fail(POLY_ERR_CUDA, std::string("cudaGetDevice: ") + cudaGetErrorString(e));
    if (dev < 0 || dev >= kMaxDevices) return fail(POLY_ERR_UNSUPPORTED, "device ordinal out of range");
    std::lock_guard<std::mutex> lk(g_setup_mu);
    if (!g_scratch_addr[dev]) {
        void* p = nullptr;
        e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
        if (e != cudaSuccess || !p)
            return fail(POLY_ERR_CUDA, std::string("cudaGetSymbolAddress: ") + cudaGetErrorString(e));
        g_scratch_addr[dev] = p;
    }
    *out = g_scratch_addr[dev];
    return POLY_OK;
}

namespace {
struct Carve {  // 256-byte aligned sub-ranges of the static array
    size_t used = 0;
    size_t take(size_t bytes) {
        const size_t off = used;
        used += (bytes + 255) / 256 * 256;
        return off;
    }
};
}  // namespace

namespace {
// The limit of this entry point, fixed so that what it takes does not move with the contraction's own
// layout: what its intermediates take with the bins cut into tiles of 64 rows (pairs (k1, k2), in the order of their
// first and last k3) by 64 columns (k3), 4096 sums per tile and split.  The buffers in use are smaller (checked below).
struct TileCount {
    size_t tiles = 0, rows = 0, cols = 0, fields = 0;
};
TileCount count_tiles(const PsPlan& p) {
    struct Row {
        int lo, hi, k1, k2;
        std::vector<int> cols;
    };
    std::vector<Row> rows;
    for (int64_t b = 0; b < p.nbins; b++) {  // bins are sorted, so a row's columns are consecutive and ascending
        const int32_t* k = &p.bins[3 * b];
        if (rows.empty() || rows.back().k1 != k[0] || rows.back().k2 != k[1]) rows.push_back({k[2], k[2], k[0], k[1], {}});
        rows.back().hi = k[2];
        rows.back().cols.push_back(k[2]);
    }
    std::stable_sort(rows.begin(), rows.end(), [](const Row& a, const Row& b) {
        return a.lo != b.lo ? a.lo < b.lo : a.hi < b.hi;
    });
    TileCount t;
    for (size_t g = 0; g < rows.size(); g += 64) {
        const size_t g1 = std::min(rows.size(), g + 64);
        std::vector<int> cu, rf;
        for (size_t r = g; r < g1; r++) {
            cu.insert(cu.end(), rows[r].cols.begin(), rows[r].cols.end());
            rf.push_back(rows[r].k1);
            rf.push_back(rows[r].k2);
        }
        std::sort(cu.begin(), cu.end());
        cu.erase(std::unique(cu.begin(), cu.end()), cu.end());
        for (size_t c0 = 0; c0 < cu.size(); c0 += 64) {
            const size_t c1 = std::min(cu.size(), c0 + 64);
            std::vector<int> f(rf);
            f.insert(f.end(), cu.begin() + (long)c0, cu.begin() + (long)c1);
            std::sort(f.begin(), f.end());
            t.tiles++;
            t.rows += g1 - g;
            t.cols += c1 - c0;
            t.fields += (size_t)(std::unique(f.begin(), f.end()) - f.begin());
        }
    }
    return t;
}
}  // namespace

static poly_status estimate_noalloc(int N, double L, int nshell, const double* edges, const float* delta_x,
                                    const int64_t* counts, double* out, void* stream) {
    if (!edges || !delta_x || !counts || !out) return fail(POLY_ERR_ARG, "NULL argument");
    if (nshell < 1 || nshell > 128) return fail(POLY_ERR_ARG, "nshell must be in [1, 128]");
    if (!(L > 0) || !std::isfinite(L)) return fail(POLY_ERR_ARG, "L must be positive");
    if (!ps_supported_n(N)) return fail(POLY_ERR_UNSUPPORTED, "grid size N not in the supported set");
    for (int s = 0; s <= nshell; s++)
        if (!std::isfinite(edges[s]) || edges[s] < 0 || (s < nshell && !(edges[s + 1] > edges[s])))
            return fail(POLY_ERR_ARG, "edges must be finite, non-negative and strictly increasing");
    const int order = 3;
    PsPlan hp;  // host-side tables only; owns no device memory
    hp.N = N;
    hp.L = L;
    hp.order = order;
    hp.nshell = nshell;
    hp.edges.assign(edges, edges + nshell + 1);
    const double emax2 = edges[nshell] * edges[nshell];
    int K = 0;
    while ((double)((long long)(K + 1) * (K + 1)) < emax2) K++;
    hp.K = K;
    if (2 * K + 1 > N) return fail(POLY_ERR_ARG, "outer shell edge exceeds the Nyquist frequency");
    if ((long long)order * K >= N) return fail(POLY_ERR_ALIAS, "3 * K >= N: triangle closures would wrap around");
    if (ps_plane_needs_spill(N, K, 0) != 0) return fail(POLY_ERR_UNSUPPORTED, "grid too large for this entry point");
    enumerate_bins(nshell, hp.edges, order, false, hp.bins);
    hp.nbins = (int64_t)hp.bins.size() / order;
    std::vector<short> lines;
    std::vector<int> line_off{0};
    for (int s = 0; s < nshell; s++) {
        build_lines(&hp, hp.edges.data(), s, lines);
        line_off.push_back((int)(lines.size() / 4));
    }
    const int64_t n3 = (int64_t)N * N * N;
    const size_t nl = (size_t)(2 * K + 1) * (K + 1);
    size_t tile_part;  // bytes of the tiles' sums
    {
        const TileCount t = count_tiles(hp);
        const int64_t nsplit = std::max<int64_t>(1, std::min<int64_t>(64, (n3 + 31) / 32 / 16));
        tile_part = (size_t)nsplit * t.tiles * 4096 * 8;
        Carve c;
        for (size_t bytes : {(size_t)N * 16, (size_t)N * 16, lines.size() * sizeof(short), line_off.size() * sizeof(int),
                             (size_t)N * nl * 8, nl * (2 * K + 1) * 8, (size_t)nshell * n3 * 4, t.tiles * 32, t.fields * 4,
                             t.rows * 8, t.cols * 8, (size_t)hp.nbins * 8, tile_part, (size_t)hp.nbins * 8,
                             (size_t)hp.nbins * 8})
            c.take(bytes);
        if (c.used > kNoAllocBytes)
            return fail(POLY_ERR_UNSUPPORTED, "this problem is over the entry point's size limit: it counts as " +
                                                  std::to_string(c.used >> 20) + " MiB, of 32 MiB");
    }
    int dev = 0, sms = 0;
    if (cudaError_t e = cudaGetDevice(&dev)) return fail(POLY_ERR_CUDA, std::string("cudaGetDevice: ") + cudaGetErrorString(e));
    if (cudaError_t e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev))
        return fail(POLY_ERR_CUDA, std::string("cudaDeviceGetAttribute: ") + cudaGetErrorString(e));
    build_cc_tasks(&hp, 0, 0, hp.cc);
    const int64_t one_row = std::max<int64_t>(1, hp.cc.ntask() * cc_span(order, false, 0, order) * 8);
    const CcLaunch cl = cc_launch_shape(hp.cc, order, nshell, n3 / 32, sms, std::max<int64_t>(1, (int64_t)tile_part / one_row));

    // layout of the static array
    Carve c;
    const size_t o_twf = c.take((size_t)N * 16), o_twi = c.take((size_t)N * 16);
    const size_t o_lines = c.take(lines.size() * sizeof(short)), o_loff = c.take(line_off.size() * sizeof(int));
    const size_t o_W = c.take((size_t)N * nl * 8), o_fhat = c.take(nl * (2 * K + 1) * 8);
    const size_t o_fields = c.take((size_t)nshell * n3 * 4);
    const size_t o_tasks = c.take(hp.cc.tasks.size() * sizeof(CcTask));
    const size_t o_groups = c.take(hp.cc.groups.size() * sizeof(CcGroup));
    const size_t o_slot = c.take(hp.cc.slot.size() * sizeof(int64_t));
    const size_t o_part = c.take((size_t)(cl.rows() * cl.stride()) * 8);
    const size_t o_cnt = c.take((size_t)hp.nbins * 8);
    if (c.used > kNoAllocBytes)
        return fail(POLY_ERR_UNSUPPORTED, "this problem needs " + std::to_string(c.used >> 20) +
                                              " MiB of scratch; the static array holds 32 MiB");

    void* base = nullptr;
    poly_status st0 = scratch_for_current_device(&base);
    if (st0) return st0;
    unsigned char* B = (unsigned char*)base;
    cudaStream_t st = (cudaStream_t)stream;

    std::vector<double> twf(2 * N), twi(2 * N);
    for (int m = 0; m < N; m++) {
        const double a = 2.0 * 3.14159265358979323846 * (double)m / (double)N;
        twf[2 * m] = std::cos(a);
        twf[2 * m + 1] = -std::sin(a);
        twi[2 * m] = std::cos(a);
        twi[2 * m + 1] = std::sin(a);
    }
    struct Copy {
        size_t off;
        const void* src;
        size_t bytes;
    } copies[] = {{o_twf, twf.data(), twf.size() * 8},
                  {o_twi, twi.data(), twi.size() * 8},
                  {o_lines, lines.data(), lines.size() * sizeof(short)},
                  {o_loff, line_off.data(), line_off.size() * sizeof(int)},
                  {o_tasks, hp.cc.tasks.data(), hp.cc.tasks.size() * sizeof(CcTask)},
                  {o_groups, hp.cc.groups.data(), hp.cc.groups.size() * sizeof(CcGroup)},
                  {o_slot, hp.cc.slot.data(), hp.cc.slot.size() * sizeof(int64_t)},
                  {o_cnt, counts, (size_t)hp.nbins * 8}};
    for (const Copy& cp : copies)
        if (cp.bytes) {
            cudaError_t e = cudaMemcpyAsync(B + cp.off, cp.src, cp.bytes, cudaMemcpyHostToDevice, st);
            if (e) return fail(POLY_ERR_CUDA, std::string("copy into scratch: ") + cudaGetErrorString(e));
        }
    const double n3d = (double)n3;
    const double norm = std::pow(L * L * L, order - 1) / std::pow(n3d, order);
    cudaError_t e;
    if ((e = ps_forward(N, 0, delta_x, K, B + o_twf, B + o_W, B + o_fhat, nullptr, st)) ||
        (e = ps_inverse(N, 0, 0, B + o_fhat, B + o_lines, (const int*)(B + o_loff), 0, nshell, K, 0, N, B + o_twi,
                        B + o_fields, (size_t)n3, nullptr, nullptr, 0, nshell, st)) ||
        (e = ps_contract_cc(0, order, 0, 0, cl, B + o_fields, nullptr, (const CcGroup*)(B + o_groups),
                            (const CcTask*)(B + o_tasks), (double*)(B + o_part), st)) ||
        (e = ps_reduce_slots((const double*)(B + o_part), (int)cl.rows(), cl.stride(), (const int64_t*)(B + o_slot),
                             (const int64_t*)(B + o_cnt), hp.nbins, norm, n3d, out, st)))
        return fail(POLY_ERR_CUDA, std::string("estimate kernels: ") + cudaGetErrorString(e));
    return POLY_OK;
}

extern "C" poly_status poly_estimate_noalloc(int N, double L, int nshell, const double* edges, const float* delta_x,
                                             const int64_t* counts, double* out, void* stream) {
    try {  // the host tables are std::vectors: no C++ exception crosses the C ABI
        return estimate_noalloc(N, L, nshell, edges, delta_x, counts, out, stream);
    } catch (const std::bad_alloc&) {
        return fail(POLY_ERR_ALLOC, "host allocation failed");
    } catch (const std::exception& ex) {
        return fail(POLY_ERR_ARG, ex.what());
    }
}
