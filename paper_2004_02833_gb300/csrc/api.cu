// The C ABI of include/rtpn.h: context life cycle, data movement and the step schedule.
#include <cuda_bf16.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <stdexcept>
#include <string>
#include <utility>

#include "rtpn_internal.h"

using namespace rtpn;

namespace {

thread_local std::string g_create_err;

int fail(rtpn_ctx* ctx, int code, const std::string& msg) {
    if (ctx)
        ctx->err = msg;
    else
        g_create_err = msg;
    return code;
}

#define CUDA_TRY(ctx, call)                                                                      \
    do {                                                                                         \
        cudaError_t e_ = (call);                                                                 \
        if (e_ != cudaSuccess)                                                                   \
            return fail(ctx, e_ == cudaErrorMemoryAllocation ? RTPN_ENOMEM : RTPN_ECUDA,         \
                        std::string(#call) + ": " + cudaGetErrorString(e_));                     \
    } while (0)

#define CHECK_LAUNCH(ctx)                                                                        \
    do {                                                                                         \
        cudaError_t e_ = cudaGetLastError();                                                     \
        if (e_ != cudaSuccess)                                                                   \
            return fail(ctx, RTPN_ECUDA, std::string("kernel launch: ") + cudaGetErrorString(e_)); \
    } while (0)

size_t dtype_size(int dtype) { return dtype == RTPN_DTYPE_F64 ? 8 : 4; }

bool valid_dtype(int d) { return d == RTPN_DTYPE_F64 || d == RTPN_DTYPE_F32; }
bool valid_where(int w) { return w == RTPN_HOST || w == RTPN_DEVICE; }

// typed dispatch on the storage precision
template <typename Fn>
void with_storage(int prec, Fn&& fn) {
    if (prec == RTPN_FP64)
        fn((double*)nullptr);
    else if (prec == RTPN_FP32)
        fn((float*)nullptr);
    else
        fn((__nv_bfloat16*)nullptr);
}

// convert `n` values of caller dtype at device pointer `in` into storage at `out`
int convert_in(rtpn_ctx* ctx, const void* in, int dtype, void* out, long long n) {
    with_storage(ctx->prec, [&](auto tag) {
        using S = std::remove_pointer_t<decltype(tag)>;
        if (dtype == RTPN_DTYPE_F64)
            launch_convert<double, S>((const double*)in, (S*)out, n, ctx->stream);
        else
            launch_convert<float, S>((const float*)in, (S*)out, n, ctx->stream);
    });
    CHECK_LAUNCH(ctx);
    return RTPN_OK;
}

int convert_out(rtpn_ctx* ctx, const void* in, void* out, int dtype, long long n) {
    with_storage(ctx->prec, [&](auto tag) {
        using S = std::remove_pointer_t<decltype(tag)>;
        if (dtype == RTPN_DTYPE_F64)
            launch_convert<S, double>((const S*)in, (double*)out, n, ctx->stream);
        else
            launch_convert<S, float>((const S*)in, (float*)out, n, ctx->stream);
    });
    CHECK_LAUNCH(ctx);
    return RTPN_OK;
}

bool same_type(int prec, int dtype) {
    return (prec == RTPN_FP64 && dtype == RTPN_DTYPE_F64) ||
           (prec == RTPN_FP32 && dtype == RTPN_DTYPE_F32);
}

void* comp_ptr(rtpn_ctx* ctx, int internal) {
    return (char*)ctx->u + (size_t)internal * ctx->sV * ctx->elem;
}

// rows between a dense array of the caller's type and the (padded) state; one component without a
// permutation, or all of them
RowCopy rows_of(const rtpn_ctx* ctx, bool into_state, bool all) {
    const Geom& g = ctx->g;
    RowCopy r{g.nx, into_state ? g.nx : ctx->px, into_state ? ctx->px : g.nx, all ? ctx->md.nc : 1,
              (long long)g.ny * g.nz, into_state ? g.V : ctx->sV, into_state ? ctx->sV : g.V,
              all ? ctx->perm : nullptr, into_state};
    return r;
}
void rows_in(rtpn_ctx* ctx, const void* in, int dtype, void* state, bool all) {
    const RowCopy r = rows_of(ctx, true, all);
    with_storage(ctx->prec, [&](auto tag) {
        using S = std::remove_pointer_t<decltype(tag)>;
        if (dtype == RTPN_DTYPE_F64)
            launch_rows<double, S>((const double*)in, (S*)state, r, ctx->stream);
        else
            launch_rows<float, S>((const float*)in, (S*)state, r, ctx->stream);
    });
}
void rows_out(rtpn_ctx* ctx, const void* state, void* out, int dtype, bool all) {
    const RowCopy r = rows_of(ctx, false, all);
    with_storage(ctx->prec, [&](auto tag) {
        using S = std::remove_pointer_t<decltype(tag)>;
        if (dtype == RTPN_DTYPE_F64)
            launch_rows<S, double>((const S*)state, (double*)out, r, ctx->stream);
        else
            launch_rows<S, float>((const S*)state, (float*)out, r, ctx->stream);
    });
}

// Whether kernels of the context may dereference the caller's device pointer: memory of the context's GPU
// (or managed), aligned for its type, with that GPU current.  Anything else (another GPU's memory, with
// or without peer access, page-locked host memory, odd addresses) goes through the runtime's copies.
bool direct(const rtpn_ctx* ctx, const void* p, int dtype) {
    cudaPointerAttributes at{};
    int dev = -1;
    if (reinterpret_cast<uintptr_t>(p) % dtype_size(dtype) != 0) return false;
    if (cudaPointerGetAttributes(&at, p) != cudaSuccess || cudaGetDevice(&dev) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    if (dev != ctx->device) return false;
    return at.type == cudaMemoryTypeManaged || (at.type == cudaMemoryTypeDevice && at.device == ctx->device);
}

int put_component(rtpn_ctx* ctx, int abi, const void* src, int dtype, int where) {
    const long long V = ctx->g.V;
    void* dst = comp_ptr(ctx, ctx->md.internal_of_abi[abi]);
    const size_t bytes = (size_t)V * dtype_size(dtype);
    const cudaMemcpyKind kind = where == RTPN_HOST ? cudaMemcpyHostToDevice : cudaMemcpyDeviceToDevice;
    if (same_type(ctx->prec, dtype) && !ctx->padded()) {
        CUDA_TRY(ctx, cudaMemcpyAsync(dst, src, bytes, kind, ctx->stream));
        return RTPN_OK;
    }
    const void* dev = src;
    if (where == RTPN_HOST || !direct(ctx, src, dtype)) {
        CUDA_TRY(ctx, cudaMemcpyAsync(ctx->staging, src, bytes, kind, ctx->stream));
        dev = ctx->staging;
    }
    if (!ctx->padded()) return convert_in(ctx, dev, dtype, dst, V);
    rows_in(ctx, dev, dtype, dst, false);
    CHECK_LAUNCH(ctx);
    return RTPN_OK;
}

int take_component(rtpn_ctx* ctx, int abi, void* dst, int dtype, int where) {
    const long long V = ctx->g.V;
    const void* src = comp_ptr(ctx, ctx->md.internal_of_abi[abi]);
    const size_t bytes = (size_t)V * dtype_size(dtype);
    const cudaMemcpyKind kind = where == RTPN_HOST ? cudaMemcpyDeviceToHost : cudaMemcpyDeviceToDevice;
    if (same_type(ctx->prec, dtype) && !ctx->padded()) {
        CUDA_TRY(ctx, cudaMemcpyAsync(dst, src, bytes, kind, ctx->stream));
        return RTPN_OK;
    }
    const bool staged = where == RTPN_HOST || !direct(ctx, dst, dtype);
    void* dev = staged ? ctx->staging : dst;
    if (ctx->padded()) {
        rows_out(ctx, src, dev, dtype, false);
        CHECK_LAUNCH(ctx);
    } else if (int rc = convert_out(ctx, src, dev, dtype, V)) {
        return rc;
    }
    if (staged) CUDA_TRY(ctx, cudaMemcpyAsync(dst, dev, bytes, kind, ctx->stream));
    return RTPN_OK;
}

// ------------------------------------------------------------------ step schedule
// whether the generic kernel has a compiled form for this FP64 context
bool generic_compiled(const rtpn_ctx* ctx) {
    return ctx->prec == RTPN_FP64 && !ctx->scat && cubic_cells(ctx->g) && window64_supported(ctx->N);
}

int run_pass(rtpn_ctx* ctx, int cls, int fac_ofs, cudaStream_t st) {
    if (ctx->active_kernel == RTPN_KERNEL_STAGE) {
        int rc = launch_stage(ctx, cls, fac_ofs, st, -1, STAGE_WAIT_LIMIT);
        if (rc) return fail(ctx, RTPN_ECUDA, std::string("staged kernel: ") +
                                                 cudaGetErrorString((cudaError_t)rc));
    } else if (ctx->active_kernel == RTPN_KERNEL_WINDOW || ctx->active_kernel == RTPN_KERNEL_FUSED) {
        WindowLaunch w;
        w.u = ctx->u;
        w.fac = (const float*)ctx->fac;
        w.g = ctx->g;
        w.cls = cls;
        w.aniso = ctx->scat != nullptr;
        w.fac_ofs = w.aniso && fac_ofs == FAC_HALF ? aniso_half_ofs(ctx->N) : fac_ofs;
        const bool own_tile = ctx->active_kernel == RTPN_KERNEL_WINDOW;
        w.tx = own_tile ? ctx->tx : 0;
        w.ty = own_tile ? ctx->ty : 0;
        w.tz = own_tile ? ctx->tz : 0;
        int rc = launch_window(ctx->N, ctx->prec, w, st);
        if (rc) return fail(ctx, RTPN_ECUDA, std::string("window kernel: ") +
                                                 cudaGetErrorString((cudaError_t)rc));
    } else if (ctx->prec == RTPN_FP64 && generic_compiled(ctx)) {
        int rc = launch_window64(ctx->N, (double*)ctx->u, (const double*)ctx->fac, ctx->g, cls, fac_ofs, st);
        if (rc) return fail(ctx, RTPN_ECUDA, std::string("generic kernel: ") + cudaGetErrorString((cudaError_t)rc));
    } else if (ctx->prec == RTPN_FP64) {
        if (ctx->scat && fac_ofs == FAC_HALF) fac_ofs = aniso_half_ofs(ctx->N);
        launch_substep_generic<double, double>((double*)ctx->u, (const double*)ctx->fac,
                                               ctx->tab64[cls], ctx->g, fac_ofs, st);
    } else if (ctx->prec == RTPN_FP32) {
        if (ctx->scat && fac_ofs == FAC_HALF) fac_ofs = aniso_half_ofs(ctx->N);
        launch_substep_generic<float, float>((float*)ctx->u, (const float*)ctx->fac,
                                             ctx->tab32[cls], ctx->g, fac_ofs, st);
    } else {
        if (ctx->scat && fac_ofs == FAC_HALF) fac_ofs = aniso_half_ofs(ctx->N);
        launch_substep_generic<__nv_bfloat16, float>((__nv_bfloat16*)ctx->u,
                                                     (const float*)ctx->fac, ctx->tab32[cls],
                                                     ctx->g, fac_ofs, st);
    }
    CHECK_LAUNCH(ctx);
    return RTPN_OK;
}

// One fused pass (even full step, odd step with factors fac_odd) from state x into state y.
int fused_pass(rtpn_ctx* ctx, const void* x, void* y, int fac_odd, cudaStream_t st) {
    FusedLaunch f;
    f.x = x;
    f.y = y;
    f.fac = (const float*)ctx->fac;
    f.g = ctx->g;
    f.fac_odd = fac_odd;
    f.zc = ctx->tz;
    int rc = launch_fused(ctx->N, ctx->prec, f, st);
    if (rc) return fail(ctx, RTPN_ECUDA, std::string("fused kernel: ") + cudaGetErrorString((cudaError_t)rc));
    return RTPN_OK;
}

void* other_buffer(const rtpn_ctx* ctx, const void* cur) { return cur == ctx->u ? ctx->u_alt : ctx->u; }

// `pairs` fused passes alternating between the two buffers, starting from state `from`; the state
// ends in `from` for an even count and in the other buffer for an odd one.
int enqueue_fused(rtpn_ctx* ctx, int pairs, void* from, cudaStream_t st) {
    void* x = from;
    for (int p = 0; p < pairs; ++p) {
        void* y = other_buffer(ctx, x);
        int rc = fused_pass(ctx, x, y, FAC_FULL, st);
        if (rc) return rc;
        x = y;
    }
    return RTPN_OK;
}

int enqueue_pairs(rtpn_ctx* ctx, int pairs, bool fused, cudaStream_t st) {
    if (fused) return enqueue_fused(ctx, pairs, ctx->u, st);
    for (int p = 0; p < pairs; ++p) {
        int rc = run_pass(ctx, 0, FAC_FULL, st);
        if (rc) return rc;
        rc = run_pass(ctx, 1, FAC_FULL, st);
        if (rc) return rc;
    }
    return RTPN_OK;
}

void drop_graphs(rtpn_ctx* ctx) {
    for (auto& kv : ctx->graphs) cudaGraphExecDestroy(kv.second);
    ctx->graphs.clear();
}

// (even, odd) full-step pairs, replayed from cached graphs of 64 / 8 / 1 pairs.  Fused passes
// alternate between the two state buffers: their graphs are keyed by which buffer they start from
// (the buffer addresses are fixed for the life of the context) and ctx->u follows the state.
// `fused` = false runs the two-pass schedule (also with RTPN_KERNEL_FUSED active).
int launch_pairs(rtpn_ctx* ctx, int pairs, bool fused) {
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    CUDA_TRY(ctx, cudaStreamIsCapturing(ctx->stream, &cap));
    if (cap != cudaStreamCaptureStatusNone) {
        int rc = enqueue_pairs(ctx, pairs, fused, ctx->stream);
        if (!rc && fused && (pairs & 1)) std::swap(ctx->u, ctx->u_alt);
        return rc;
    }
    const int sizes[3] = {64, 8, 1};
    for (int s : sizes) {
        while (pairs >= s) {
            // key: pair count, plus 1 << 20 for fused graphs starting from the second buffer
            const int key = fused ? s + (1 << 16) + (ctx->u == ctx->u_home ? 0 : 1 << 20) : s;
            auto it = ctx->graphs.find(key);
            if (it == ctx->graphs.end()) {
                cudaGraph_t graph = nullptr;
                CUDA_TRY(ctx, cudaStreamBeginCapture(ctx->own, cudaStreamCaptureModeThreadLocal));
                int rc = enqueue_pairs(ctx, s, fused, ctx->own);
                cudaError_t e = cudaStreamEndCapture(ctx->own, &graph);
                if (rc) {
                    if (graph) cudaGraphDestroy(graph);
                    return rc;
                }
                if (e != cudaSuccess)
                    return fail(ctx, RTPN_ECUDA, std::string("capture: ") + cudaGetErrorString(e));
                cudaGraphExec_t exec = nullptr;
                e = cudaGraphInstantiate(&exec, graph, 0);
                cudaGraphDestroy(graph);
                if (e != cudaSuccess)
                    return fail(ctx, RTPN_ECUDA, std::string("instantiate: ") + cudaGetErrorString(e));
                it = ctx->graphs.emplace(key, exec).first;
            }
            CUDA_TRY(ctx, cudaGraphLaunch(it->second, ctx->stream));
            if (fused && (s & 1)) std::swap(ctx->u, ctx->u_alt);
            pairs -= s;
        }
    }
    return RTPN_OK;
}

HostTable host_table(const Model& md, int cls, const Geom& g, bool aniso) {
    HostTable t;
    t.a0 = cls == 0 ? 0 : md.ne;
    t.na = cls == 0 ? md.ne : md.no;
    t.row.push_back(0);
    // md.nz is sorted by row (interface index); targets come in internal order, so index rows first
    std::vector<size_t> first(md.nc + 1, md.nz.size());
    for (size_t q = md.nz.size(); q-- > 0;) first[md.nz[q].a] = q;
    for (int i = t.a0; i < t.a0 + t.na; ++i) {
        const int a = md.abi_of_internal[i];
        const Component& ca = md.comp[a];
        for (size_t q = first[a]; q < md.nz.size() && md.nz[q].a == a; ++q) {
            const Coupling& e = md.nz[q];
            const bool upper = ca.slot[e.axis] == 2;  // target on a 2-slot reads cells i, i+1
            t.src.push_back(md.internal_of_abi[e.b]);
            t.code.push_back(e.axis * 2 + (upper ? 1 : 0));
            t.coef.push_back((upper ? 1.0 : -1.0) * e.v / axis_h(g, e.axis));
        }
        t.row.push_back((int)t.src.size());
        t.fplane.push_back(a == 0 ? FAC_U0
                                  : aniso ? aniso_plane(md.N, slot_code(ca.slot), ca.l) : 2 * slot_code(ca.slot));
    }
    return t;
}

// upload both classes' tables into one allocation (ints, then doubles, then floats)
int upload_tables(rtpn_ctx* ctx) {
    const bool aniso = ctx->scat != nullptr;
    HostTable t[2] = {host_table(ctx->md, 0, ctx->g, aniso), host_table(ctx->md, 1, ctx->g, aniso)};
    size_t bytes = 0;
    for (auto& x : t)
        bytes += (x.row.size() + x.src.size() + x.code.size() + x.fplane.size()) * sizeof(int) +
                 x.coef.size() * (sizeof(double) + sizeof(float)) + 64;
    CUDA_TRY(ctx, cudaMalloc(&ctx->table_mem, bytes));
    std::vector<char> host(bytes, 0);
    size_t off = 0;
    auto put = [&](const void* src, size_t n) {
        off = (off + 7) & ~size_t(7);
        std::memcpy(host.data() + off, src, n);
        size_t at = off;
        off += n;
        return (char*)ctx->table_mem + at;
    };
    for (int c = 0; c < 2; ++c) {
        auto& x = t[c];
        std::vector<float> cf(x.coef.begin(), x.coef.end());
        const int* row = (const int*)put(x.row.data(), x.row.size() * sizeof(int));
        const int* src = (const int*)put(x.src.data(), x.src.size() * sizeof(int));
        const int* code = (const int*)put(x.code.data(), x.code.size() * sizeof(int));
        const int* fp = (const int*)put(x.fplane.data(), x.fplane.size() * sizeof(int));
        const double* c64 = (const double*)put(x.coef.data(), x.coef.size() * sizeof(double));
        const float* c32 = (const float*)put(cf.data(), cf.size() * sizeof(float));
        ctx->tab64[c] = {row, src, c64, code, fp, x.a0, x.na};
        ctx->tab32[c] = {row, src, c32, code, fp, x.a0, x.na};
    }
    CUDA_TRY(ctx, cudaMemcpy(ctx->table_mem, host.data(), bytes, cudaMemcpyHostToDevice));
    return RTPN_OK;
}

void release(rtpn_ctx* ctx) {
    drop_graphs(ctx);
    if (ctx->u) cudaFree(ctx->u);
    if (ctx->u_alt) cudaFree(ctx->u_alt);
    ctx->u_alt = ctx->u_home = nullptr;
    if (ctx->fac) cudaFree(ctx->fac);
    if (ctx->scat) cudaFree(ctx->scat);
    ctx->scat = nullptr;
    if (ctx->table_mem) cudaFree(ctx->table_mem);
    if (ctx->perm) cudaFree(ctx->perm);
    ctx->perm = nullptr;
    if (ctx->partial) cudaFree(ctx->partial);
    if (ctx->counter) cudaFree(ctx->counter);
    if (ctx->staging) cudaFree(ctx->staging);
    if (ctx->status) cudaFree(ctx->status);
    if (ctx->media) cudaFree(ctx->media);
    ctx->media = nullptr;
    if (ctx->stage_mem) cudaFree(ctx->stage_mem);
    if (ctx->stage_maps_dev) cudaFree(ctx->stage_maps_dev);
    ctx->stage_maps_dev = nullptr;
    if (ctx->adj_ws) cudaFree(ctx->adj_ws);
    ctx->adj_ws = nullptr;
    ctx->adj_ws_bytes = 0;
    for (long long& k : ctx->adj_maps_key) k = -1;
    ctx->status = nullptr;
    ctx->stage_mem = nullptr;
    if (ctx->own) cudaStreamDestroy(ctx->own);
    ctx->u = ctx->fac = ctx->table_mem = ctx->staging = nullptr;
    ctx->partial = nullptr;
    ctx->counter = nullptr;
    ctx->own = nullptr;
}

// Automatic selection: the staged kernel where it is compiled for (N, precision) and N >= kStageMinN, on
// padded rows where nx does not give 16-byte ones, else the register-window kernel, else the generic
// one.  Padding costs at most three (FP32) or seven (BF16) columns of traffic; the kernels that take any
// width cost far more there (GB300, FP32, a pass: P15 61 x 77 x 75 0.14 ms against
// 0.24 on the window kernel, P19 0.18 against 1.09 on the generic one, P39 0.68 against 3.25 on the window
// kernel).  Below kStageMinN the unrolled window body is small enough for the instruction cache and the
// staged kernel's barriers and copies per stage weigh more (P7 128^3: 0.36 ms a step with the window
// kernel, 0.38 with the staged one).
constexpr bool kStageInAuto = true;
constexpr int kStageMinN = 15;
// Rows of fewer than 8 cells are not padded: up to three cells in four would be padding, and the staged tiles
// are at least 32 cells wide.  (GB300, us a step on n x n x nx cells, staged / the kernel it replaces: P15 window
// kernel, n = 12, 24, 48: nx = 9 30 / 52, 32 / 54, 37 / 59; nx = 33 29 / 56, 35 / 59, 88 / 123; P39 window kernel:
// nx = 9 114 / 232, 119 / 223, 390 / 816.  P19 and P29 run the generic kernel otherwise, whose targets are split over
// blocks on small grids: below some 5000 cells it is the faster one (P19 nx = 9: 41 / 18, 44 / 38, 91 / 117; P29 nx = 33
// 69 / 70, 88 / 251), though far from the 650 us such a P19 step took before the split.)
constexpr int kPadMinNx = 8;

// Row pitch of the state: nx, or nx padded to 16-byte rows.  set_rows rearranges the state in place, a component
// at a time through the staging plane (its buffer holds the padded state if the context can ever need
// it); the padding holds zeros.
int padded_pitch(const rtpn_ctx* ctx) {
    return stage_row_pitch(ctx->prec, ctx->g.nx);
}
int set_rows(rtpn_ctx* ctx, int px) {
    const Geom& g = ctx->g;
    if (px == ctx->px) return RTPN_OK;
    const long long sV = (long long)px * g.ny * g.nz, rows = (long long)g.ny * g.nz;
    drop_graphs(ctx);
    for (int k = 0; k < ctx->md.nc; ++k) {
        const int c = px > ctx->px ? ctx->md.nc - 1 - k : k;  // growing: from the last component
        with_storage(ctx->prec, [&](auto tag) {
            using S = std::remove_pointer_t<decltype(tag)>;
            if constexpr (!std::is_same_v<S, double>) {  // FP64 states are never padded
                const S* from = (const S*)ctx->u + (size_t)c * ctx->sV;
                S* to = (S*)ctx->u + (size_t)c * sV;
                launch_rows<S, S>(from, (S*)ctx->staging, RowCopy{g.nx, ctx->px, g.nx, 1, rows, 0, 0, nullptr, true}, ctx->stream);
                launch_rows<S, S>((const S*)ctx->staging, to, RowCopy{g.nx, g.nx, px, 1, rows, 0, 0, nullptr, true}, ctx->stream);
            }
        });
    }
    ctx->px = px;
    ctx->sV = sV;
    CHECK_LAUNCH(ctx);
    return RTPN_OK;
}

// whether the automatic choice may pad the rows for the staged kernel
bool may_pad(const rtpn_ctx* ctx) {
    return kStageInAuto && ctx->N >= kStageMinN && !ctx->batch_member && !ctx->no_padding && ctx->g.nx >= kPadMinNx &&
           stage_compiled(ctx->N, ctx->prec) && stage_sized(ctx->prec, ctx->g);
}

// The kernel for the context's selection, with what it needs.  Whatever can fail comes first; the kernel, its
// tile and the rows of the state then change together, so a failure leaves the context as it was.
int choose_kernel(rtpn_ctx* ctx) {
    int k = ctx->kernel;
    int tx = ctx->tx, ty = ctx->ty, tz = ctx->tz, depth = ctx->depth;
    bool from_stage = ctx->tile_from_stage;
    const bool cubic = cubic_cells(ctx->g);
    if (ctx->scat) {
        // per-order factors: the generic kernel's per-target plane table, or the window kernel's
        // anisotropic form (N <= 15), which reads each target's planes at its finish
        const bool win_aniso = window_supported(ctx->N, ctx->prec) && window_extended(ctx->N);
        if (k == RTPN_KERNEL_AUTO) k = win_aniso ? RTPN_KERNEL_WINDOW : RTPN_KERNEL_GENERIC;
        if (k != RTPN_KERNEL_GENERIC && !(k == RTPN_KERNEL_WINDOW && win_aniso))
            return fail(ctx, RTPN_EUNSUPPORTED,
                        "anisotropic scattering runs on the generic kernel and the window kernel up to N = 15");
    }
    // the window kernel takes non-cubic cells up to N = 15 (scaled y and z differences); the fused
    // kernel takes cubic cells only
    const bool win_ok = window_supported(ctx->N, ctx->prec) && (cubic || window_extended(ctx->N));
    if (k == RTPN_KERNEL_AUTO) {
        const bool tile_set = (tx || ty || tz) && !from_stage;
        // other widths than 16-byte rows: padded, unless the caller asks for a tile, or for a stage depth that
        // no variant has (then one of the kernels that take any width)
        const bool pad = may_pad(ctx) && !ctx->dense_rows && !tile_set &&
                         stage_has_tile(ctx->N, tx, ty, tz, depth, ctx->prec);
        if (kStageInAuto && (ctx->N >= kStageMinN || !win_ok) &&
            (stage_supported(ctx->N, ctx->prec, ctx->g) || pad) &&
            (!tile_set || stage_has_tile(ctx->N, tx, ty, tz, depth, ctx->prec)))
            k = RTPN_KERNEL_STAGE;
        else
            k = win_ok ? RTPN_KERNEL_WINDOW : RTPN_KERNEL_GENERIC;
    }
    // a tile the staged kernel chose is no request for another kernel (its shape need not even be a
    // valid window tile): the other kernels start from their defaults
    if (k != RTPN_KERNEL_STAGE && from_stage) {
        tx = ty = tz = depth = 0;
        from_stage = false;
    }
    if (!cubic && k == RTPN_KERNEL_FUSED)
        return fail(ctx, RTPN_EUNSUPPORTED, "the fused kernel takes cubic cells only");
    if (!cubic && k == RTPN_KERNEL_WINDOW && !window_extended(ctx->N))
        return fail(ctx, RTPN_EUNSUPPORTED, "the window kernel takes non-cubic cells up to N = 15 only");
    // the automatic choice runs the staged kernel on any width of rows, padding them; chosen by name it
    // takes 16-byte rows only
    const bool pad = k == RTPN_KERNEL_STAGE && ctx->kernel == RTPN_KERNEL_AUTO &&
                     !stage_supported(ctx->N, ctx->prec, ctx->g);
    if (k == RTPN_KERNEL_STAGE && !pad) {
        if (!stage_supported(ctx->N, ctx->prec, ctx->g))
            return fail(ctx, RTPN_EUNSUPPORTED,
                        "staged kernel not compiled for this N/precision, nx*elem not 16-byte rows or a component of 4 GiB");
        if (!stage_has_tile(ctx->N, tx, ty, tz, depth, ctx->prec))
            return fail(ctx, RTPN_EUNSUPPORTED, "no staged kernel compiled for this tile / stage depth");
    }
    auto unprepared = [&](const char* what, int rc) {
        cudaGetLastError();  // reported here; the next launch check is not to see it
        return fail(ctx,
                    rc == (int)cudaErrorMemoryAllocation ? RTPN_ENOMEM
                    : rc == (int)cudaErrorNotSupported   ? RTPN_EUNSUPPORTED
                                                         : RTPN_ECUDA,
                    std::string(what) + ": " + cudaGetErrorString((cudaError_t)rc));
    };
    const int px = pad ? padded_pitch(ctx) : ctx->g.nx;
    if (px != ctx->px) {
        // recorded into the caller's graph, the rearranging would run at each replay and not now
        cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
        if (cudaStreamIsCapturing(ctx->stream, &cap) != cudaSuccess || cap != cudaStreamCaptureStatusNone) {
            cudaGetLastError();
            return fail(ctx, RTPN_ESTATE, "the state's rows cannot be rearranged while the stream is being captured");
        }
    }
    if (k == RTPN_KERNEL_GENERIC && generic_compiled(ctx)) {
        int rc = window64_prepare(ctx->md);
        if (rc) return unprepared("generic kernel constants", rc);
    }
    if (k == RTPN_KERNEL_WINDOW) {
        if (!window_supported(ctx->N, ctx->prec))
            return fail(ctx, RTPN_EUNSUPPORTED, "window kernel not compiled for this N/precision");
        int rc = window_prepare(ctx->md, ctx->g.h, ctx->prec);
        if (rc) return unprepared("window constants", rc);
    }
    if (k == RTPN_KERNEL_FUSED) {
        // a batch keeps each instance's state pointer in its launch items; the fused kernel moves it
        if (ctx->batch_member)
            return fail(ctx, RTPN_EUNSUPPORTED, "batch instances keep their state in one buffer");
        if (!fused_supported(ctx->N, ctx->prec) || !window_supported(ctx->N, ctx->prec))
            return fail(ctx, RTPN_EUNSUPPORTED, "fused kernel not compiled for this N/precision");
        int rc = fused_prepare(ctx->md, ctx->prec);
        if (!rc) rc = window_prepare(ctx->md, ctx->g.h, ctx->prec);
        if (rc) return unprepared("fused kernel constants", rc);
        if (!ctx->u_alt) {
            cudaError_t e = cudaMalloc(&ctx->u_alt, (size_t)ctx->md.nc * ctx->g.V * ctx->elem);
            if (e != cudaSuccess) {
                ctx->u_alt = nullptr;
                cudaGetLastError();
                return fail(ctx, RTPN_ENOMEM, "second state buffer of the fused kernel");
            }
        }
    }
    if (k == RTPN_KERNEL_STAGE) {
        int rc = stage_prepare(ctx, tx, ty, tz, depth, px);  // sets the tile
        if (rc) return unprepared("staged kernel set-up", rc);
    } else {
        ctx->tx = tx;
        ctx->ty = ty;
        ctx->tz = tz;
        ctx->depth = depth;
        ctx->tile_from_stage = from_stage;
    }
    if (k != ctx->active_kernel) drop_graphs(ctx);
    ctx->active_kernel = k;
    return set_rows(ctx, px);
}

}  // namespace

namespace rtpn {
// Message for rtpn_last_error(NULL) from entry points that take no context.
void note_error(const std::string& msg) { g_create_err = msg; }
}  // namespace rtpn

// ==================================================================== C ABI
extern "C" {

int rtpn_version(void) { return 100; }

const char* rtpn_strerror(int code) {
    switch (code) {
        case RTPN_OK: return "ok";
        case RTPN_EINVAL: return "invalid argument";
        case RTPN_ECFL: return "time step violates dt < min(h)/3";
        case RTPN_ENOMEM: return "device allocation failed";
        case RTPN_ECUDA: return "CUDA error";
        case RTPN_ETIMEOUT: return "bounded device wait expired";
        case RTPN_ENONFINITE: return "non-finite values in the state";
        case RTPN_EUNSUPPORTED: return "not compiled into this library";
        case RTPN_ESTATE: return "call out of order";
        default: return "unknown status";
    }
}

int rtpn_component_info(int N, int c, int* l, int* m, int slots[3], int* cls) {
    if (N < 0 || N > 63 || c < 0 || c >= (N + 1) * (N + 1)) return RTPN_EINVAL;
    int L = 0;
    while ((L + 1) * (L + 1) <= c) ++L;
    const int mm = c - L * L - L;
    const int M = mm < 0 ? -mm : mm;
    const int t = mm < 0 ? 1 : 0;
    const int sgnM = (M % 2 == 0) ? 1 : -1;
    const int px = t == 0 ? sgnM : -sgnM, py = t == 0 ? 1 : -1, pz = ((L + M) % 2 == 0) ? 1 : -1;
    if (l) *l = L;
    if (m) *m = mm;
    if (slots) {
        slots[0] = px == 1 ? 1 : 2;
        slots[1] = py == 1 ? 1 : 2;
        slots[2] = pz == 1 ? 1 : 2;
    }
    if (cls) *cls = L % 2;
    return RTPN_OK;
}

int rtpn_coupling_dense(int N, int axis, double* out) {
    if (N < 0 || N > 63 || axis < 0 || axis > 2 || !out) return RTPN_EINVAL;
    Model md = build_model(N);
    const size_t n = md.nc;
    std::memset(out, 0, n * n * sizeof(double));
    for (const auto& e : md.nz)
        if (e.axis == axis) out[(size_t)e.a * n + e.b] = e.v;
    return RTPN_OK;
}

int rtpn_create(rtpn_ctx** out, int N, int nx, int ny, int nz, double h, int bc, int precision,
                double dt) {
    return rtpn::create_context(out, N, nx, ny, nz, h, bc, precision, dt, false);
}

}  // extern "C"

int rtpn::use_staged_tile(rtpn_ctx* ctx, int tx, int ty, int tz, int depth) {
    if (!ctx->padded() || !stage_has_tile(ctx->N, tx, ty, tz, depth, ctx->prec))
        return fail(ctx, RTPN_EUNSUPPORTED, "no staged kernel compiled for this tile / stage depth");
    const int ox = ctx->tx, oy = ctx->ty, oz = ctx->tz, oc = ctx->depth;
    drop_graphs(ctx);
    ctx->tx = tx;
    ctx->ty = ty;
    ctx->tz = tz;
    ctx->depth = depth;
    const int rc = choose_kernel(ctx);  // the selection is AUTO and tile_from_stage stays set
    if (rc) {
        ctx->tx = ox;
        ctx->ty = oy;
        ctx->tz = oz;
        ctx->depth = oc;
    }
    return rc;
}

int rtpn::use_dense_rows(rtpn_ctx* ctx, bool on) {
    if (ctx->dense_rows == on) return RTPN_OK;
    const int tile[4] = {ctx->tx, ctx->ty, ctx->tz, ctx->depth};
    ctx->dense_rows = on;
    int rc = choose_kernel(ctx);
    if (rc) {
        ctx->dense_rows = !on;
        return rc;
    }
    if (on)
        std::copy(tile, tile + 4, ctx->padded_tile);
    else if (ctx->padded())
        rc = use_staged_tile(ctx, ctx->padded_tile[0], ctx->padded_tile[1], ctx->padded_tile[2], ctx->padded_tile[3]);
    return rc;
}

namespace {
// create_context with or without room for padded rows
int create_with(rtpn_ctx** out, int N, int nx, int ny, int nz, double h, int bc, int precision, double dt, bool batch_member,
                bool pad, bool* padded) {
    if (!out) return fail(nullptr, RTPN_EINVAL, "out is NULL");
    *out = nullptr;
    if (N < 0 || N > 63) return fail(nullptr, RTPN_EINVAL, "N must be in 0..63");
    if (nx < 1 || ny < 1 || nz < 1) return fail(nullptr, RTPN_EINVAL, "grid dims must be >= 1");
    if (!(h > 0.0) || !std::isfinite(h)) return fail(nullptr, RTPN_EINVAL, "h must be > 0");
    if (bc != RTPN_BC_PERIODIC && bc != RTPN_BC_VACUUM)
        return fail(nullptr, RTPN_EINVAL, "unknown boundary");
    if (precision != RTPN_FP64 && precision != RTPN_FP32 && precision != RTPN_BF16)
        return fail(nullptr, RTPN_EINVAL, "unknown precision");
    if (dt <= 0.0) dt = 0.3 * h;
    if (!(dt < h / 3.0)) return fail(nullptr, RTPN_ECFL, "dt must be below h/3 (Section 2.1)");
    const long long V = (long long)nx * ny * nz;
    if (V > (1ll << 40)) return fail(nullptr, RTPN_EINVAL, "grid too large");

    rtpn_ctx* ctx = new rtpn_ctx();
    ctx->md = build_model(N);
    ctx->N = N;
    ctx->g = Geom{nx, ny, nz, V, bc, h, h, h};
    ctx->prec = precision;
    ctx->dt = dt;
    ctx->batch_member = batch_member;
    ctx->no_padding = !pad;
    ctx->px = nx;
    ctx->sV = V;
    ctx->elem = precision == RTPN_FP64 ? 8 : (precision == RTPN_FP32 ? 4 : 2);
    const size_t fac_elem = precision == RTPN_FP64 ? 8 : 4;
    auto bail = [&](int rc) {
        g_create_err = ctx->err;
        release(ctx);
        delete ctx;
        return rc;
    };
    int rc;
    if (cudaGetDevice(&ctx->device) != cudaSuccess) return bail(fail(ctx, RTPN_ECUDA, "no CUDA device"));
    if (cudaStreamCreateWithFlags(&ctx->own, cudaStreamDefault) != cudaSuccess)
        return bail(fail(ctx, RTPN_ECUDA, "stream create failed"));
    ctx->stream = ctx->own;
    // room for padded rows where the automatic choice may take them
    const int room_px = may_pad(ctx) ? padded_pitch(ctx) : nx;
    *padded = room_px != nx;
    const size_t state_room = (size_t)ctx->md.nc * room_px * ny * nz * ctx->elem;
    cudaError_t e = cudaMalloc(&ctx->u, state_room);
    if (e != cudaSuccess) return bail(fail(ctx, RTPN_ENOMEM, "state allocation failed"));
    ctx->u_home = ctx->u;
    e = cudaMalloc(&ctx->fac, (size_t)FAC_PLANES * V * fac_elem);
    if (e != cudaSuccess) return bail(fail(ctx, RTPN_ENOMEM, "factor allocation failed"));
    e = cudaMalloc(&ctx->staging, (size_t)V * 8);
    if (e != cudaSuccess) return bail(fail(ctx, RTPN_ENOMEM, "staging allocation failed"));
    e = cudaMalloc(&ctx->perm, ctx->md.nc * sizeof(int));
    if (e != cudaSuccess) return bail(fail(ctx, RTPN_ENOMEM, "scratch allocation failed"));
    e = cudaMemcpy(ctx->perm, ctx->md.internal_of_abi.data(), ctx->md.nc * sizeof(int), cudaMemcpyHostToDevice);
    if (e != cudaSuccess) return bail(fail(ctx, RTPN_ECUDA, cudaGetErrorString(e)));
    e = cudaMalloc(&ctx->partial, (SUM_BLOCKS + 1) * sizeof(double));
    if (e != cudaSuccess) return bail(fail(ctx, RTPN_ENOMEM, "scratch allocation failed"));
    e = cudaMalloc(&ctx->counter, sizeof(unsigned long long));
    if (e != cudaSuccess) return bail(fail(ctx, RTPN_ENOMEM, "scratch allocation failed"));
    e = cudaMalloc(&ctx->status, 10 * sizeof(unsigned));
    if (e != cudaSuccess) return bail(fail(ctx, RTPN_ENOMEM, "status allocation failed"));
    ctx->tickets = ctx->status + 8;
    e = cudaMemsetAsync(ctx->status, 0, 10 * sizeof(unsigned), ctx->stream);
    if (e != cudaSuccess) return bail(fail(ctx, RTPN_ECUDA, cudaGetErrorString(e)));
    if ((rc = upload_tables(ctx))) return bail(rc);
    e = cudaMemsetAsync(ctx->u, 0, state_room, ctx->stream);
    if (e != cudaSuccess) return bail(fail(ctx, RTPN_ECUDA, cudaGetErrorString(e)));
    // a state of zeros needs no rearranging: padded from the start where the choice below pads it
    ctx->px = room_px;
    ctx->sV = (long long)room_px * ny * nz;
    if ((rc = choose_kernel(ctx))) return bail(rc);
    e = cudaStreamSynchronize(ctx->stream);
    if (e != cudaSuccess) return bail(fail(ctx, RTPN_ECUDA, cudaGetErrorString(e)));
    *out = ctx;
    return RTPN_OK;
}
}  // namespace

int rtpn::create_context(rtpn_ctx** out, int N, int nx, int ny, int nz, double h, int bc, int precision, double dt,
                         bool batch_member) {
    bool padded = false;
    int rc = create_with(out, N, nx, ny, nz, h, bc, precision, dt, batch_member, true, &padded);
    if (rc == RTPN_ENOMEM && padded) {  // the padding must not be what keeps a problem off the device
        cudaGetLastError();
        rc = create_with(out, N, nx, ny, nz, h, bc, precision, dt, batch_member, false, &padded);
    }
    return rc;
}

extern "C" {

int rtpn_destroy(rtpn_ctx* ctx) {
    if (!ctx) return RTPN_OK;
    if (ctx->stream) cudaStreamSynchronize(ctx->stream);
    release(ctx);
    delete ctx;
    return RTPN_OK;
}

}  // extern "C"

namespace {
// The tables that a call replaces, put back if a later part of it fails: the context is then as it was, and its
// kernels have tables to read.
struct KeptTables {
    rtpn_ctx* c;
    void *mem, *stage = nullptr;
    bool with_stage;
    size_t stage_bytes[2];
    PartnerTable<double> t64[2];
    PartnerTable<float> t32[2];
    KeptTables(rtpn_ctx* ctx, bool with_staged) : c(ctx), mem(ctx->table_mem), with_stage(with_staged) {
        for (int i = 0; i < 2; ++i) {
            t64[i] = c->tab64[i];
            t32[i] = c->tab32[i];
            stage_bytes[i] = c->stage_tab_bytes[i];
        }
        c->table_mem = nullptr;
        if (with_stage) std::swap(stage, c->stage_mem);
    }
    void put_back() {
        if (c->table_mem) cudaFree(c->table_mem);
        c->table_mem = mem;
        for (int i = 0; i < 2; ++i) {
            c->tab64[i] = t64[i];
            c->tab32[i] = t32[i];
        }
        if (with_stage) {
            if (c->stage_mem) cudaFree(c->stage_mem);
            c->stage_mem = stage;
            std::copy(stage_bytes, stage_bytes + 2, c->stage_tab_bytes);
        }
    }
    void drop() {
        if (mem) cudaFree(mem);
        if (stage) cudaFree(stage);
    }
};
}  // namespace

extern "C" {

int rtpn_set_spacing(rtpn_ctx* ctx, double hx, double hy, double hz) {
    if (!ctx) return RTPN_EINVAL;
    if (!(hx > 0.0 && hy > 0.0 && hz > 0.0) || !std::isfinite(hx) || !std::isfinite(hy) ||
        !std::isfinite(hz))
        return fail(ctx, RTPN_EINVAL, "cell sizes must be positive and finite");
    if (!(ctx->dt < std::min(hx, std::min(hy, hz)) / 3.0))
        return fail(ctx, RTPN_ECFL, "dt must be below min(hx, hy, hz)/3 (Section 2.1)");
    const bool cubic = hx == hy && hy == hz;
    // a batch keeps each instance's 1/h in its launch items, built at creation
    if (ctx->batch_member)
        return fail(ctx, RTPN_EUNSUPPORTED, "the spacing of a batch instance is fixed at creation");
    const Geom old = ctx->g;
    ctx->g.h = hx;
    ctx->g.hy = hy;
    ctx->g.hz = hz;
    auto restore = [&](int code, const std::string& msg) {
        ctx->g = old;
        return fail(ctx, code, msg);
    };
    if (!cubic && (ctx->kernel == RTPN_KERNEL_FUSED ||
                   (ctx->kernel == RTPN_KERNEL_WINDOW && !window_extended(ctx->N))))
        return restore(RTPN_EUNSUPPORTED, "the fused kernel, and the window kernel above N = 15, take cubic cells only");
    // the partner tables and the staged kernel's constants carry the spacing: rebuild them
    if (cudaError_t e = cudaStreamSynchronize(ctx->stream)) return restore(RTPN_ECUDA, cudaGetErrorString(e));
    drop_graphs(ctx);
    KeptTables kept(ctx, true);
    int rc = upload_tables(ctx);
    if (!rc) rc = choose_kernel(ctx);
    if (rc) {
        cudaGetLastError();
        kept.put_back();
        ctx->g = old;
        return rc;
    }
    kept.drop();
    return RTPN_OK;
}

int rtpn_set_scattering(rtpn_ctx* ctx, const double* f, int count) {
    if (!ctx) return RTPN_EINVAL;
    const bool iso = f == nullptr || count == 0;
    if (!iso) {
        if (count != ctx->N + 1) return fail(ctx, RTPN_EINVAL, "give f_0 .. f_N (count = N + 1)");
        if (f[0] != 1.0) return fail(ctx, RTPN_EINVAL, "f_0 must be 1 (Sigma_s0 = sigma_s)");
        for (int l = 1; l <= ctx->N; ++l)
            if (!(f[l] >= -1.0 && f[l] <= 1.0)) return fail(ctx, RTPN_EINVAL, "f_l must lie in [-1, 1]");
        if (ctx->batch_member)
            return fail(ctx, RTPN_EUNSUPPORTED, "batch instances take isotropic scattering only");
        const bool win_aniso = window_supported(ctx->N, ctx->prec) && window_extended(ctx->N);
        if (ctx->kernel != RTPN_KERNEL_AUTO && ctx->kernel != RTPN_KERNEL_GENERIC &&
            !(ctx->kernel == RTPN_KERNEL_WINDOW && win_aniso))
            return fail(ctx, RTPN_EUNSUPPORTED,
                        "anisotropic scattering runs on the generic kernel and the window kernel up to N = 15");
    }
    CUDA_TRY(ctx, cudaStreamSynchronize(ctx->stream));
    const long long V = ctx->g.V;
    const size_t fac_elem = ctx->prec == RTPN_FP64 ? 8 : 4;
    const int planes = iso ? FAC_PLANES : aniso_planes(ctx->N);
    // new buffers first, so that a failed allocation leaves the context as it was
    double* scat = nullptr;
    void* fac = nullptr;
    if (!iso) {
        cudaError_t e = cudaMalloc(&scat, sizeof(double) * (ctx->N + 1));
        if (e == cudaSuccess) e = cudaMemcpy(scat, f, sizeof(double) * (ctx->N + 1), cudaMemcpyHostToDevice);
        if (e != cudaSuccess) {
            if (scat) cudaFree(scat);
            cudaGetLastError();
            return fail(ctx, RTPN_ENOMEM, "scattering moments");
        }
    }
    if (planes != ctx->fac_planes) {
        cudaError_t e = cudaMalloc(&fac, (size_t)planes * V * fac_elem);
        if (e != cudaSuccess) {
            if (scat) cudaFree(scat);
            cudaGetLastError();
            return fail(ctx, RTPN_ENOMEM, "factor planes of anisotropic scattering");
        }
    }
    drop_graphs(ctx);
    double* const old_scat = ctx->scat;
    void* const old_fac = ctx->fac;
    const int old_planes = ctx->fac_planes;
    ctx->scat = scat;
    if (fac) {
        ctx->fac = fac;
        ctx->fac_planes = planes;
    }
    KeptTables kept(ctx, false);
    int rc = upload_tables(ctx);
    if (!rc) rc = choose_kernel(ctx);
    if (rc) {
        cudaGetLastError();
        kept.put_back();
        if (scat) cudaFree(scat);
        if (fac) cudaFree(fac);
        ctx->scat = old_scat;
        ctx->fac = old_fac;
        ctx->fac_planes = old_planes;
        return rc;
    }
    kept.drop();
    if (old_scat) cudaFree(old_scat);
    if (fac) cudaFree(old_fac);
    if (ctx->media_set) {  // the factors of the media already set, with the new moments
        const double* m = ctx->media;
        if (ctx->prec == RTPN_FP64)
            launch_media_factors<double>(m, m + V, m + 2 * V, (double*)ctx->fac, ctx->g, ctx->dt,
                                         ctx->scat, ctx->N, ctx->stream);
        else
            launch_media_factors<float>(m, m + V, m + 2 * V, (float*)ctx->fac, ctx->g, ctx->dt,
                                        ctx->scat, ctx->N, ctx->stream);
        CUDA_TRY(ctx, cudaGetLastError());
        CUDA_TRY(ctx, cudaStreamSynchronize(ctx->stream));
    }
    return rc;
}

int rtpn_set_stream(rtpn_ctx* ctx, void* stream) {
    if (!ctx) return RTPN_EINVAL;
    ctx->stream = stream ? (cudaStream_t)stream : ctx->own;
    return RTPN_OK;
}

int rtpn_set_kernel(rtpn_ctx* ctx, int kernel, int tile_x, int tile_y, int tile_z) {
    return rtpn_set_kernel_ex(ctx, kernel, tile_x, tile_y, tile_z, 0);
}

int rtpn_set_kernel_ex(rtpn_ctx* ctx, int kernel, int tile_x, int tile_y, int tile_z, int depth) {
    if (!ctx) return RTPN_EINVAL;
    if (depth < 0 || depth > 8) return fail(ctx, RTPN_EINVAL, "bad stage depth");
    if (kernel < RTPN_KERNEL_AUTO || kernel > RTPN_KERNEL_FUSED)
        return fail(ctx, RTPN_EINVAL, "unknown kernel");
    if (tile_x < 0 || tile_y < 0 || tile_z < 0) return fail(ctx, RTPN_EINVAL, "bad tile");
    if (kernel == RTPN_KERNEL_FUSED) {
        if ((tile_x && tile_x != 32) || (tile_y && tile_y != 8))
            return fail(ctx, RTPN_EINVAL, "the fused kernel's tile is 32 x 8 cells");
    } else if (kernel != RTPN_KERNEL_STAGE && (tile_x || tile_y || tile_z)) {
        const long long th = (long long)(tile_x ? tile_x : 32) * (tile_y ? tile_y : 4) *
                             (tile_z ? tile_z : 2);
        if (th > 256 || th % 32 != 0)
            return fail(ctx, RTPN_EINVAL, "tile must hold a multiple of 32 threads, at most 256");
    }
    const int old = ctx->kernel, ox = ctx->tx, oy = ctx->ty, oz = ctx->tz, oc = ctx->depth;
    const bool ofs = ctx->tile_from_stage;
    ctx->kernel = kernel;
    drop_graphs(ctx);
    ctx->tx = tile_x;
    ctx->ty = tile_y;
    ctx->tz = tile_z;
    ctx->tile_from_stage = false;
    ctx->depth = kernel == RTPN_KERNEL_STAGE || kernel == RTPN_KERNEL_AUTO ? depth : 0;
    int rc = choose_kernel(ctx);
    if (rc) {  // nothing has changed but the selection
        ctx->kernel = old;
        ctx->tx = ox;
        ctx->ty = oy;
        ctx->tz = oz;
        ctx->depth = oc;
        ctx->tile_from_stage = ofs;
    }
    return rc;
}

int rtpn_set_media(rtpn_ctx* ctx, const void* sigma_a, const void* sigma_s, const void* q,
                   int dtype, int where) {
    if (!ctx || !sigma_a || !sigma_s || !q) return RTPN_EINVAL;
    if (!valid_dtype(dtype) || !valid_where(where)) return fail(ctx, RTPN_EINVAL, "bad dtype/where");
    const long long V = ctx->g.V;
    // the FP64 media stay on the device (the adjoint needs them again)
    if (!ctx->media) CUDA_TRY(ctx, cudaMalloc(&ctx->media, (size_t)3 * V * sizeof(double)));
    double* m = ctx->media;
    const void* srcs[3] = {sigma_a, sigma_s, q};
    const size_t bytes = (size_t)V * dtype_size(dtype);
    int rc = RTPN_OK;
    for (int i = 0; i < 3 && !rc; ++i) {
        double* dst = m + (size_t)i * V;
        const void* src = srcs[i];
        cudaError_t e = cudaSuccess;
        if (dtype == RTPN_DTYPE_F64) {
            e = cudaMemcpyAsync(dst, src, bytes,
                                where == RTPN_HOST ? cudaMemcpyHostToDevice
                                                   : cudaMemcpyDeviceToDevice,
                                ctx->stream);
        } else {
            if (where == RTPN_HOST) {
                e = cudaMemcpyAsync(ctx->staging, src, bytes, cudaMemcpyHostToDevice, ctx->stream);
                src = ctx->staging;
            }
            if (e == cudaSuccess) launch_convert<float, double>((const float*)src, dst, V, ctx->stream);
        }
        if (e != cudaSuccess) rc = fail(ctx, RTPN_ECUDA, cudaGetErrorString(e));
    }
    if (!rc) {
        if (ctx->prec == RTPN_FP64)
            launch_media_factors<double>(m, m + V, m + 2 * V, (double*)ctx->fac, ctx->g, ctx->dt,
                                         ctx->scat, ctx->N, ctx->stream);
        else
            launch_media_factors<float>(m, m + V, m + 2 * V, (float*)ctx->fac, ctx->g, ctx->dt,
                                        ctx->scat, ctx->N, ctx->stream);
        cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) rc = fail(ctx, RTPN_ECUDA, cudaGetErrorString(e));
    }
    cudaError_t e = cudaStreamSynchronize(ctx->stream);
    if (rc) return rc;
    if (e != cudaSuccess) return fail(ctx, RTPN_ECUDA, cudaGetErrorString(e));
    ctx->media_set = true;
    return RTPN_OK;
}

int rtpn_set_component(rtpn_ctx* ctx, int c, const void* field, int dtype, int where) {
    if (!ctx || !field) return RTPN_EINVAL;
    if (c < 0 || c >= ctx->md.nc) return fail(ctx, RTPN_EINVAL, "component out of range");
    if (!valid_dtype(dtype) || !valid_where(where)) return fail(ctx, RTPN_EINVAL, "bad dtype/where");
    int rc = put_component(ctx, c, field, dtype, where);
    if (rc) return rc;
    ctx->steps_done = 0;
    if (where == RTPN_HOST) CUDA_TRY(ctx, cudaStreamSynchronize(ctx->stream));
    return RTPN_OK;
}

int rtpn_get_component(rtpn_ctx* ctx, int c, void* field, int dtype, int where) {
    if (!ctx || !field) return RTPN_EINVAL;
    if (c < 0 || c >= ctx->md.nc) return fail(ctx, RTPN_EINVAL, "component out of range");
    if (!valid_dtype(dtype) || !valid_where(where)) return fail(ctx, RTPN_EINVAL, "bad dtype/where");
    int rc = take_component(ctx, c, field, dtype, where);
    if (rc) return rc;
    if (where == RTPN_HOST) CUDA_TRY(ctx, cudaStreamSynchronize(ctx->stream));
    return RTPN_OK;
}

int rtpn_set_moments(rtpn_ctx* ctx, const void* u, int dtype, int where) {
    if (!ctx || !u) return RTPN_EINVAL;
    if (!valid_dtype(dtype) || !valid_where(where)) return fail(ctx, RTPN_EINVAL, "bad dtype/where");
    const bool near = where == RTPN_DEVICE && direct(ctx, u, dtype);
    if (near && ctx->padded()) {
        rows_in(ctx, u, dtype, ctx->u, true);
        CHECK_LAUNCH(ctx);
        ctx->steps_done = 0;
        return RTPN_OK;
    }
    if (near) {
        with_storage(ctx->prec, [&](auto tag) {
            using S = std::remove_pointer_t<decltype(tag)>;
            if (dtype == RTPN_DTYPE_F64)
                launch_reorder<double, S>((const double*)u, (S*)ctx->u, ctx->perm, ctx->md.nc, ctx->g.V, true, ctx->stream);
            else
                launch_reorder<float, S>((const float*)u, (S*)ctx->u, ctx->perm, ctx->md.nc, ctx->g.V, true, ctx->stream);
        });
        CHECK_LAUNCH(ctx);
        ctx->steps_done = 0;
        return RTPN_OK;
    }
    const size_t plane = (size_t)ctx->g.V * dtype_size(dtype);
    for (int c = 0; c < ctx->md.nc; ++c) {
        int rc = put_component(ctx, c, (const char*)u + (size_t)c * plane, dtype, where);
        if (rc) return rc;
    }
    ctx->steps_done = 0;
    if (where == RTPN_HOST) CUDA_TRY(ctx, cudaStreamSynchronize(ctx->stream));
    return RTPN_OK;
}

int rtpn_get_moments(rtpn_ctx* ctx, void* u, int dtype, int where) {
    if (!ctx || !u) return RTPN_EINVAL;
    if (!valid_dtype(dtype) || !valid_where(where)) return fail(ctx, RTPN_EINVAL, "bad dtype/where");
    const bool near = where == RTPN_DEVICE && direct(ctx, u, dtype);
    if (near && ctx->padded()) {
        rows_out(ctx, ctx->u, u, dtype, true);
        CHECK_LAUNCH(ctx);
        return RTPN_OK;
    }
    if (near) {
        with_storage(ctx->prec, [&](auto tag) {
            using S = std::remove_pointer_t<decltype(tag)>;
            if (dtype == RTPN_DTYPE_F64)
                launch_reorder<S, double>((const S*)ctx->u, (double*)u, ctx->perm, ctx->md.nc, ctx->g.V, false, ctx->stream);
            else
                launch_reorder<S, float>((const S*)ctx->u, (float*)u, ctx->perm, ctx->md.nc, ctx->g.V, false, ctx->stream);
        });
        CHECK_LAUNCH(ctx);
        return RTPN_OK;
    }
    const size_t plane = (size_t)ctx->g.V * dtype_size(dtype);
    for (int c = 0; c < ctx->md.nc; ++c) {
        int rc = take_component(ctx, c, (char*)u + (size_t)c * plane, dtype, where);
        if (rc) return rc;
    }
    if (where == RTPN_HOST) CUDA_TRY(ctx, cudaStreamSynchronize(ctx->stream));
    return RTPN_OK;
}

int rtpn_zero_moments(rtpn_ctx* ctx) {
    if (!ctx) return RTPN_EINVAL;
    CUDA_TRY(ctx, cudaMemsetAsync(ctx->u, 0, (size_t)ctx->md.nc * ctx->sV * ctx->elem, ctx->stream));
    ctx->steps_done = 0;
    return RTPN_OK;
}

int rtpn_step(rtpn_ctx* ctx, int k) {
    if (!ctx || k < 0) return RTPN_EINVAL;
    if (!ctx->media_set) return fail(ctx, RTPN_ESTATE, "rtpn_set_media has not been called");
    if (k == 0) return RTPN_OK;
    bool fused = ctx->active_kernel == RTPN_KERNEL_FUSED;
    if (fused) {
        // a caller's capture keeps the pointers it saw: the two-pass schedule stays in one buffer
        cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
        CUDA_TRY(ctx, cudaStreamIsCapturing(ctx->stream, &cap));
        fused = cap == cudaStreamCaptureStatusNone;
    }
    int rc = run_pass(ctx, 1, FAC_HALF, ctx->stream);
    if (!rc) rc = launch_pairs(ctx, k - 1, fused);
    if (fused) {
        if (!rc) rc = fused_pass(ctx, ctx->u, ctx->u_alt, FAC_HALF, ctx->stream);
        if (!rc) std::swap(ctx->u, ctx->u_alt);
    } else {
        if (!rc) rc = run_pass(ctx, 0, FAC_FULL, ctx->stream);
        if (!rc) rc = run_pass(ctx, 1, FAC_HALF, ctx->stream);
    }
    if (!rc) ctx->steps_done += k;
    return rc;
}

int rtpn_substep(rtpn_ctx* ctx, int cls, int half) {
    if (!ctx || cls < 0 || cls > 1 || half < 0 || half > 1) return RTPN_EINVAL;
    if (cls == 0 && half) return fail(ctx, RTPN_EINVAL, "the even class has no half-step factors");
    if (!ctx->media_set) return fail(ctx, RTPN_ESTATE, "rtpn_set_media has not been called");
    return run_pass(ctx, cls, half ? FAC_HALF : FAC_FULL, ctx->stream);
}

int rtpn_copy_planes(rtpn_ctx* dst, int dst_z, rtpn_ctx* src, int src_z, int nz, int cls) {
    if (!dst || !src || nz < 0 || cls < -1 || cls > 1) return RTPN_EINVAL;
    if (src->N != dst->N || src->prec != dst->prec || src->g.nx != dst->g.nx || src->g.ny != dst->g.ny)
        return fail(dst, RTPN_EINVAL, "copy_planes: the contexts differ in order, precision, nx or ny");
    if (src_z < 0 || dst_z < 0 || src_z + nz > src->g.nz || dst_z + nz > dst->g.nz)
        return fail(dst, RTPN_EINVAL, "copy_planes: planes outside a grid");
    if (src == dst && nz > 0 && src_z < dst_z + nz && dst_z < src_z + nz)
        return fail(dst, RTPN_EINVAL, "copy_planes: overlapping planes of one context");
    if (nz == 0) return RTPN_OK;
    // the components of a class are contiguous in the internal order (class 0 first)
    const int c0 = cls == 1 ? dst->md.ne : 0;
    const int n = cls == -1 ? dst->md.nc : (cls == 0 ? dst->md.ne : dst->md.no);
    auto at = [&](const rtpn_ctx* c, int comp, int z) {
        return (char*)c->u + ((size_t)comp * c->sV + (size_t)z * c->px * c->g.ny) * c->elem;
    };
    // the copy runs on dst's stream after src's queued work, and src's later work runs after it
    cudaEvent_t ev = nullptr;
    if (src->stream != dst->stream) {
        CUDA_TRY(dst, cudaEventCreateWithFlags(&ev, cudaEventDisableTiming));
        CUDA_TRY(dst, cudaEventRecord(ev, src->stream));
        CUDA_TRY(dst, cudaStreamWaitEvent(dst->stream, ev, 0));
    }
    cudaError_t e = cudaSuccess;
    if (src->px == dst->px)
        e = cudaMemcpy2DAsync(at(dst, c0, dst_z), (size_t)dst->sV * dst->elem, at(src, c0, src_z), (size_t)src->sV * src->elem,
                              (size_t)nz * dst->px * dst->g.ny * dst->elem, (size_t)n, cudaMemcpyDeviceToDevice, dst->stream);
    else  // one of the states has padded rows
        for (int c = c0; c < c0 + n && e == cudaSuccess; ++c)
            e = cudaMemcpy2DAsync(at(dst, c, dst_z), (size_t)dst->px * dst->elem, at(src, c, src_z), (size_t)src->px * src->elem,
                                  (size_t)dst->g.nx * dst->elem, (size_t)nz * dst->g.ny, cudaMemcpyDeviceToDevice, dst->stream);
    if (ev) {
        if (e == cudaSuccess) e = cudaEventRecord(ev, dst->stream);
        if (e == cudaSuccess) e = cudaStreamWaitEvent(src->stream, ev, 0);
        cudaEventDestroy(ev);
    }
    if (e != cudaSuccess) return fail(dst, RTPN_ECUDA, std::string("copy_planes: ") + cudaGetErrorString(e));
    return RTPN_OK;
}

int rtpn_sum_u0(rtpn_ctx* ctx, double* out) {
    if (!ctx || !out) return RTPN_EINVAL;
    const void* u0 = comp_ptr(ctx, ctx->md.internal_of_abi[0]);
    with_storage(ctx->prec, [&](auto tag) {
        using S = std::remove_pointer_t<decltype(tag)>;
        launch_sum<S>((const S*)u0, ctx->sV, ctx->partial, SUM_BLOCKS, ctx->partial + SUM_BLOCKS,
                      ctx->stream);
    });
    CHECK_LAUNCH(ctx);
    CUDA_TRY(ctx, cudaMemcpyAsync(out, ctx->partial + SUM_BLOCKS, sizeof(double),
                                  cudaMemcpyDeviceToHost, ctx->stream));
    CUDA_TRY(ctx, cudaStreamSynchronize(ctx->stream));
    return RTPN_OK;
}

int rtpn_count_nonfinite(rtpn_ctx* ctx, long long* out) {
    if (!ctx || !out) return RTPN_EINVAL;
    with_storage(ctx->prec, [&](auto tag) {
        using S = std::remove_pointer_t<decltype(tag)>;
        launch_count_nonfinite<S>((const S*)ctx->u, (long long)ctx->md.nc * ctx->sV, ctx->counter,
                                  ctx->stream);
    });
    CHECK_LAUNCH(ctx);
    unsigned long long c = 0;
    CUDA_TRY(ctx, cudaMemcpyAsync(&c, ctx->counter, sizeof(c), cudaMemcpyDeviceToHost, ctx->stream));
    CUDA_TRY(ctx, cudaStreamSynchronize(ctx->stream));
    *out = (long long)c;
    return c ? fail(ctx, RTPN_ENONFINITE, "non-finite values in the state") : RTPN_OK;
}

int rtpn_synchronize(rtpn_ctx* ctx) {
    if (!ctx) return RTPN_EINVAL;
    CUDA_TRY(ctx, cudaStreamSynchronize(ctx->stream));
    unsigned st[8] = {0, 0, 0, 0, 0, 0, 0, 0};
    CUDA_TRY(ctx, cudaMemcpy(st, ctx->status, sizeof(st), cudaMemcpyDeviceToHost));
    if (st[0]) {
        std::string rec;
        for (int i = 0; i < 8; ++i) rec += (i ? " " : "") + std::to_string(st[i]);
        CUDA_TRY(ctx, cudaMemset(ctx->status, 0, sizeof(st)));
        if (st[0] & 1u)
            return fail(ctx, RTPN_ETIMEOUT, "a bounded wait in a staged kernel ran out [" + rec + "]");
        return fail(ctx, RTPN_ECUDA, "a staged-kernel self-check failed [" + rec + "]");
    }
    CUDA_TRY(ctx, cudaMemset(ctx->status, 0, sizeof(st)));
    return RTPN_OK;
}

int rtpn_test_wait_timeout(rtpn_ctx* ctx, int cls, long long wait_limit) {
    if (!ctx || cls < 0 || cls > 1 || wait_limit < 1) return RTPN_EINVAL;
    if (ctx->active_kernel != RTPN_KERNEL_STAGE)
        return fail(ctx, RTPN_EUNSUPPORTED, "the staged kernel is not active");
    if (!ctx->media_set) return fail(ctx, RTPN_ESTATE, "rtpn_set_media has not been called");
    // stage 1 of every CTA's sequence is never issued
    int rc = launch_stage(ctx, cls, FAC_FULL, ctx->stream, 1, wait_limit);
    if (rc) return fail(ctx, RTPN_ECUDA, cudaGetErrorString((cudaError_t)rc));
    return RTPN_OK;
}

int rtpn_get_info(const rtpn_ctx* ctx, rtpn_info* out) {
    if (!ctx || !out) return RTPN_EINVAL;
    out->N = ctx->N;
    out->n_c = ctx->md.nc;
    out->n_even = ctx->md.ne;
    out->n_odd = ctx->md.no;
    out->nx = ctx->g.nx;
    out->ny = ctx->g.ny;
    out->nz = ctx->g.nz;
    out->bc = ctx->g.bc;
    out->precision = ctx->prec;
    out->kernel = ctx->active_kernel;
    out->h = ctx->g.h;
    out->hy = ctx->g.hy;
    out->hz = ctx->g.hz;
    out->dt = ctx->dt;
    out->state_bytes = (size_t)ctx->md.nc * ctx->sV * ctx->elem;
    out->factor_bytes = (size_t)ctx->fac_planes * ctx->g.V * (ctx->prec == RTPN_FP64 ? 8 : 4);
    out->steps_done = ctx->steps_done;
    out->tile[0] = ctx->tx;
    out->tile[1] = ctx->ty;
    out->tile[2] = ctx->tz;
    out->depth = ctx->active_kernel == RTPN_KERNEL_STAGE ? ctx->depth : 1;
    return RTPN_OK;
}

const char* rtpn_last_error(const rtpn_ctx* ctx) {
    return ctx ? ctx->err.c_str() : g_create_err.c_str();
}

}  // extern "C"
