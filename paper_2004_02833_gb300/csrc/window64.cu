// The generic kernel's compiled form for FP64 at low orders: the register-window body (window_impl.cuh) in
// double arithmetic.
//
// An FP64 pass is bound by the FP64 rate (about 0.6 T fused multiply-adds a second on a GB300).  The
// partner-table kernel takes a difference and a product for every (target, partner) pair, about 17
// operations a source; the window body takes each source's three differences once and at most ten
// products, 12 on average, with no index loads.  GB300, without -> with: P3 32^3, forty steps with the state
// out, 534 -> 419 us; P7 64^3 0.29 / 0.31 -> 0.20 / 0.20 ms an even / odd pass.  Orders up to 9, cubic cells,
// isotropic scattering; the table kernel takes the rest.
#include <mutex>
#include <set>
#include <utility>

#include "window_impl.cuh"

#define RTPN_ORDERS64(X) X(1) X(3) X(5) X(7) X(9)

namespace rtpn {
namespace {

#define RTPN_CONST64(n)                                                    \
    __constant__ double c_coef_##n##_0[win::class_size(n, 1) * 10];        \
    __constant__ double c_coef_##n##_1[win::class_size(n, 0) * 10];
RTPN_ORDERS64(RTPN_CONST64)
#undef RTPN_CONST64

template <int N, int A>
__device__ __forceinline__ const double* coef_of() {
#define RTPN_CASE(n) \
    if constexpr (N == n) return A == 0 ? c_coef_##n##_0 : c_coef_##n##_1;
    RTPN_ORDERS64(RTPN_CASE)
#undef RTPN_CASE
    return nullptr;
}

// The launch over a grid: a.tx > 0, tiles of 32 cells of a row (times 1 x 1 or 2 x 2 rows); a.tx = 0, the cells in
// the order of memory, so that short rows share a warp.  An FP64-bound warp costs the same with one lane
// as with 32: tiles only where they keep nine lanes in ten.  (GB300, P7 64 x 64 x nx, a step in us, the table
// kernel / tiles / this: nx = 5 128 / 212 / 48, 16 188 / 212 / 114, 33 376 / 421 / 216, 65 648 / 626 / 424.)  One warp per block until every SM has eight
// 128-thread blocks: the FP64 units of every SM then have about the same number of warps to serve.
void shape64(const Geom& g, win::Args* a, unsigned* blocks, unsigned* threads) {
    const bool small = g.V < 152ll * 8 * 128;
    const int row = (g.nx + 31) / 32 * 32;
    if (10ll * g.nx >= 9ll * row) {
        a->tx = 32;
        a->ty = a->tz = small ? 1 : 2;
        a->ntx = (g.nx + a->tx - 1) / a->tx;
        a->nty = (g.ny + a->ty - 1) / a->ty;
        a->ntz = (g.nz + a->tz - 1) / a->tz;
        *blocks = (unsigned)a->ntx * a->nty * a->ntz;
        *threads = (unsigned)(a->tx * a->ty * a->tz);
    } else {
        a->tx = a->ty = a->tz = a->ntx = a->nty = a->ntz = 0;
        *threads = small ? 32 : 128;
        *blocks = (unsigned)((g.V + *threads - 1) / *threads);
    }
}
RTPN_HD bool cell64(const win::Args& a, unsigned blk, unsigned tid, unsigned threads, int* x, int* y, int* z) {
    if (a.tx > 0) return win::cell_of(a, (int)blk, (int)tid, x, y, z);
    const long long c = (long long)blk * threads + tid;
    if (c >= a.V) return false;
    // 32-bit divisions where they do (a 64-bit one is tens of instructions)
    const long long row = a.V < (1ll << 32) ? (long long)((unsigned)c / (unsigned)a.nx) : c / a.nx;
    *x = (int)(c - row * a.nx);
    *z = a.V < (1ll << 32) ? (int)((unsigned)row / (unsigned)a.ny) : (int)(row / a.ny);
    *y = (int)(row - (long long)*z * a.ny);
    return true;
}

template <int N, int A>
__global__ void __launch_bounds__(128) k_window64(win::Args a) {
    int x, y, z;
    if (!cell64(a, blockIdx.x, threadIdx.x, blockDim.x, &x, &y, &z)) return;
    win::substep_cell<N, A, double, false, false, double>(a, coef_of<N, A>(), x, y, z);
}

}  // namespace

bool window64_supported(int N) {
    switch (N) {
#define RTPN_CASE(n) case n:
        RTPN_ORDERS64(RTPN_CASE)
#undef RTPN_CASE
        return true;
        default:
            return false;
    }
}

int window64_prepare(const Model& md) {
    static std::mutex mu;
    static std::set<std::pair<int, int>> done;  // (N, device)
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return (int)e;
    std::lock_guard<std::mutex> lock(mu);
    if (done.count({md.N, dev})) return 0;
    for (int A = 0; A < 2; ++A) {
        std::vector<double> t;
        if (!win::coef_table(md, A, &t)) return (int)cudaErrorInvalidValue;
        switch (md.N) {
#define RTPN_CASE(n)                                                                                             \
    case n:                                                                                                      \
        e = A == 0 ? cudaMemcpyToSymbol(c_coef_##n##_0, t.data(), t.size() * sizeof(double))                     \
                   : cudaMemcpyToSymbol(c_coef_##n##_1, t.data(), t.size() * sizeof(double));                    \
        break;
            RTPN_ORDERS64(RTPN_CASE)
#undef RTPN_CASE
            default:
                return (int)cudaErrorNotSupported;
        }
        if (e != cudaSuccess) return (int)e;
    }
    done.insert({md.N, dev});
    return 0;
}

int launch_window64(int N, double* u, const double* fac, const Geom& g, int cls, int fac_ofs, cudaStream_t st) {
    win::Args a;
    a.u = u;
    a.fac = reinterpret_cast<const float*>(fac);  // read as FP64 by the FP64 body
    a.V = g.V;
    a.nx = g.nx;
    a.ny = g.ny;
    a.nz = g.nz;
    a.bc = g.bc;
    a.fac_ofs = fac_ofs;
    a.inv_h = (float)(1.0 / g.h);
    a.inv_h64 = 1.0 / g.h;
    unsigned blocks, threads;
    shape64(g, &a, &blocks, &threads);
    switch (N) {
#define RTPN_CASE(n)                                                  \
    case n:                                                           \
        if (cls == 0)                                                 \
            k_window64<n, 0><<<blocks, threads, 0, st>>>(a);          \
        else                                                          \
            k_window64<n, 1><<<blocks, threads, 0, st>>>(a);          \
        break;
        RTPN_ORDERS64(RTPN_CASE)
#undef RTPN_CASE
        default:
            return (int)cudaErrorNotSupported;
    }
    return (int)cudaGetLastError();
}

}  // namespace rtpn
