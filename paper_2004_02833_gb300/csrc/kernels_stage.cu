// Host side of the TMA-staged kernels: variant registry, tensor maps, coupling tables, launch.
#include <cudaTypedefs.h>

#include <cmath>
#include <mutex>
#include <numeric>
#include <vector>

#include "stage_impl.cuh"
#include "stage_variants.h"

namespace rtpn {
namespace stg {

#define RTPN_SDECL1(n, x, y, z, b, e, f)                                                                     \
    int stage_launch_##n##_##x##_##y##_##z##_##b##_##e##_##f(int, int, int, const Args&, int, cudaStream_t);  \
    int stage_smem_##n##_##x##_##y##_##z##_##b##_##e##_##f(int, int);                                          \
    void stage_geom_##n##_##x##_##y##_##z##_##b##_##e##_##f(int, int*);
#define RTPN_SDECL(n, x, y, z, b, e) RTPN_SDECL1(n, x, y, z, b, e, 0) RTPN_SDECL1(n, x, y, z, b, e, 1)
RTPN_STAGE_VARIANTS(RTPN_SDECL)
#undef RTPN_SDECL
#undef RTPN_SDECL1

struct Variant {
    int N, tx, ty, tz, depth, substages;
    // by form: 0 plain, 1 SC (h_y != h_x)
    int (*launch[2])(int, int, int, const Args&, int, cudaStream_t);  // (cls, precision, mode, ...)
    int (*smem)(int, int);
    void (*geom[2])(int, int*);  // (precision, {maps per kind, CTAs per SM, x group width, x group rows})
};
#define RTPN_SNAME(a, n, x, y, z, b, e, f) a##_##n##_##x##_##y##_##z##_##b##_##e##_##f
#define RTPN_SENTRY(n, x, y, z, b, e)                                                                                 \
    Variant{n, x, y, z, b, e, {RTPN_SNAME(stage_launch, n, x, y, z, b, e, 0), RTPN_SNAME(stage_launch, n, x, y, z, b, e, 1)}, \
            RTPN_SNAME(stage_smem, n, x, y, z, b, e, 0),                                                              \
            {RTPN_SNAME(stage_geom, n, x, y, z, b, e, 0), RTPN_SNAME(stage_geom, n, x, y, z, b, e, 1)}},
static const Variant kVariants[] = {RTPN_STAGE_VARIANTS(RTPN_SENTRY)};
#undef RTPN_SENTRY
#undef RTPN_SNAME

static int form_of(const rtpn::Geom& g) { return g.hy != g.h ? 1 : 0; }

// a variant is usable for a storage precision if its stage ring fits shared memory (of both forms or of neither)
static bool fits(const Variant& v, int precision) { return v.smem(0, precision) > 0 && v.smem(1, precision) > 0; }

// first compiled variant of order N with this tile (0 = any) and depth (0 = any) that fits
static const Variant* find(int N, int tx, int ty, int tz, int depth, int precision) {
    for (const auto& v : kVariants)
        if (v.N == N && (tx == 0 || (v.tx == tx && v.ty == ty && v.tz == tz)) &&
            (depth == 0 || v.depth == depth) && fits(v, precision))
            return &v;
    return nullptr;
}

static PFN_cuTensorMapEncodeTiled_v12000 encode_fn() {
    static std::once_flag once;
    static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
    std::call_once(once, [] {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
    });
    return fn;
}

// px, sV: row pitch and component stride of the array.  The map spans the padding of padded rows too: it holds zeros,
// as the columns outside the map would read.
static bool make_map(CUtensorMap* m, void* base, int precision, const rtpn::Geom& g, int px, long long sV, int nc,
                     int bx, int by, int bz, int bc) {
    auto fn = encode_fn();
    if (!fn) return false;
    const cuuint64_t es = precision == RTPN_BF16 ? 2 : 4;
    const cuuint64_t dims[4] = {(cuuint64_t)px, (cuuint64_t)g.ny, (cuuint64_t)g.nz, (cuuint64_t)nc};
    const cuuint64_t strides[3] = {px * es, (cuuint64_t)px * g.ny * es, (cuuint64_t)sV * es};
    const cuuint32_t box[4] = {(cuuint32_t)bx, (cuuint32_t)by, (cuuint32_t)bz, (cuuint32_t)bc};
    const cuuint32_t estr[4] = {1, 1, 1, 1};
    CUresult r = fn(m, precision == RTPN_BF16 ? CU_TENSOR_MAP_DATA_TYPE_BFLOAT16 : CU_TENSOR_MAP_DATA_TYPE_FLOAT32,
                    4, base, dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                    CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS;
}

// The tensor maps of one array for a variant (kinds MAP_PLANE, MAP_YROW, MAP_XGRP, each for box
// lengths E = 1, 2, ..., nmap; see stage_impl.cuh) into out[0 .. kinds * nmap); kinds = 1 builds the
// plane maps only (target arrays).
static bool make_maps(CUtensorMap* out, void* base, int precision, const rtpn::Geom& g, int px, long long sV, int nc,
                      const Variant& v, int kinds) {
    int geo[4];
    v.geom[0](precision, geo);
    const int nmap = geo[0], xw = geo[2], ry = geo[3];
    for (int j = 0; j < nmap; ++j) {
        const int e = j + 1;
        if (!make_map(&out[MAP_PLANE * nmap + j], base, precision, g, px, sV, nc, v.tx, v.ty, 1, e)) return false;
        if (kinds > 1 && (!make_map(&out[MAP_YROW * nmap + j], base, precision, g, px, sV, nc, v.tx, 1, v.tz, e) ||
                          !make_map(&out[MAP_XGRP * nmap + j], base, precision, g, px, sV, nc, xw, ry, v.tz, e)))
            return false;
    }
    return true;
}

// The default variant for a grid: the one whose tiles cover it at the least cost, rounds of the persistent
// CTAs times the cost of a round.  Padding at the grid's edges and an emptier last round cost as much as
// full tiles.  A round costs its cells per SM plus a fixed part in cells: the issue of a stage's boxes and its
// barriers (90 with the seven boxes a type of a two-plane tile), above order 30 also the latency of a warp's
// own instructions (400 in all).  Rows off the 128-byte lines touch more lines than they fill; half of that
// excess is felt.  GB300, FP32, a round: P15 96^3 13.2 us with two CTAs of 32x2x2, 17.1 with one of 96x2x2,
// 23.8 with one of 32x4x4 (0.303, 0.274 and 0.286 ms a pass; P19 80^3 0.246 ms with 80x2x2, 0.289 with two CTAs
// of 40x2x2); P39 69 us with 192 cells, 82 with 320, and 32x3x3 tiles 82 us at 96^3 (aligned), 113 at 120^3.
// Measured on FP32 grids at N = 15, 19 and 39; N = 29, N = 7 and BF16 take the constants over.  Against every variant by
// name on 18 grids of 320 to 262144 cells (N = 15 to 39, both storages) the choice is within 5 % of the best but at P15
// (up to 18 % on grids of one or two rounds) and, at P29 and P39 near one round, where it was the one-stage variants
// that it no longer takes.
static const Variant* best_variant(int N, int precision, int depth, const rtpn::Geom& g, int px, int sms) {
    const Variant* best = nullptr;
    double best_cost = 0;
    // From N = 29 on a tile's stages one after another are most of a small grid's pass, and columns in one stage of
    // 15 or 20 slots take longer than in sub-stages, whatever the rounds: such variants run by name only.  GB300,
    // us a step, 32x2x2 in one stage / in two: P39 FP32 20x22x32 143 / 117, 40x43x32 387 / 320, BF16 183 / 145, 400 / 338;
    // P29 FP32 80 / 69, BF16 90 / 80.
    const bool sub_staged = N >= 29;
    const int es = precision == RTPN_BF16 ? 2 : 4;
    for (const auto& v : kVariants) {
        if (v.N != N || (depth != 0 && v.depth != depth) || !fits(v, precision)) continue;
        if (sub_staged && depth == 0 && v.substages == 1) continue;
        int geo[4];
        v.geom[form_of(g)](precision, geo);
        const long long tiles = (long long)((g.nx + v.tx - 1) / v.tx) * ((g.ny + v.ty - 1) / v.ty) * ((g.nz + v.tz - 1) / v.tz);
        const long long slots = (long long)sms * geo[1];
        const long long rounds = (tiles + slots - 1) / slots;
        // a grid of less than a round leaves SMs with fewer CTAs than they hold
        const long long per_sm = rounds > 1 ? geo[1] : (tiles + sms - 1) / sms;
        const double fixed = (N > 30 ? 400.0 : 90.0) * (2 * v.tz + 3) / 7;
        const int row = v.tx * es, align = std::gcd(std::gcd(row, px * es), 128);
        const double lines = 1.0 + 0.5 * (128 - align) / row;  // row / 128 lines filled, (128 - align) / 128 more touched
        const double cost = rounds * (per_sm * v.tx * v.ty * v.tz * lines + fixed);
        if (!best || cost < best_cost) {
            best = &v;
            best_cost = cost;
        }
    }
    return best;
}

static int nmaps_of(const Variant& v, int precision) {
    int geo[4];
    v.geom[0](precision, geo);
    return geo[0];
}

}  // namespace stg

// device tensor-map slots of a context: forward (all kinds), adjoint w (all kinds), adjoint lam (plane)
static constexpr int stage_maps_capacity = (2 * stg::MAP_KINDS + 1) * stg::kMaxSlots;

bool stage_compiled(int N, int precision) {
    return precision != RTPN_FP64 && stg::find(N, 0, 0, 0, 0, precision) != nullptr;
}

bool stage_sized(int precision, const Geom& g) {
    const int px = g.nx % stage_row_group(precision) == 0 ? g.nx : stage_row_pitch(precision, g.nx);
    return (long long)px * g.ny * g.nz < (1ll << 32) / (precision == RTPN_BF16 ? 2 : 4);
}

bool stage_supported(int N, int precision, const Geom& g) {
    return stage_compiled(N, precision) && g.nx % stage_row_group(precision) == 0 && stage_sized(precision, g);
}

// stages of a pass over the grid, at most: the kernel counts a CTA's in 32 bits
static long long stages_of(const stg::Variant& v, const Geom& g) {
    return (long long)((g.nx + v.tx - 1) / v.tx) * ((g.ny + v.ty - 1) / v.ty) * ((g.nz + v.tz - 1) / v.tz) * (v.N + 2) *
           v.substages;
}

bool stage_has_tile(int N, int tx, int ty, int tz, int depth, int precision) {
    return stg::find(N, tx, ty, tz, depth, precision) != nullptr;
}

int stage_prepare(rtpn_ctx* ctx, int tx, int ty, int tz, int depth, int px) {
    const stg::Variant* v = stg::find(ctx->N, tx, ty, tz, depth, ctx->prec);
    if (!v) return (int)cudaErrorNotSupported;
    int dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&ctx->sms, cudaDevAttrMultiProcessorCount, dev);
    if (tx == 0)
        if (const stg::Variant* w = stg::best_variant(ctx->N, ctx->prec, depth, ctx->g, px, ctx->sms)) v = w;
    if (stages_of(*v, ctx->g) >= (1ll << 31)) return (int)cudaErrorNotSupported;
    const int N = ctx->N;
    // the tensor maps live in device global memory (64-byte aligned) and the kernel reads them from
    // there: tile planes / z halo plane, y halo row and x halo group, each for every box length
    const int nmap = stg::nmaps_of(*v, ctx->prec);
    if (nmap <= 0 || nmap > stg::kMaxSlots) return (int)cudaErrorInvalidValue;
    std::vector<CUtensorMap> maps((size_t)stg::MAP_KINDS * nmap);
    if (!stg::make_maps(maps.data(), ctx->u, ctx->prec, ctx->g, px, (long long)px * ctx->g.ny * ctx->g.nz, ctx->md.nc, *v,
                        stg::MAP_KINDS))
        return (int)cudaErrorInvalidValue;
    if (!ctx->stage_maps_dev) {
        // the forward's maps, then room for the adjoint's (all kinds over w, plane maps over lam)
        cudaError_t err = cudaMalloc(&ctx->stage_maps_dev, stage_maps_capacity * sizeof(CUtensorMap));
        if (err != cudaSuccess) return (int)err;
    }
    if (!ctx->stage_mem) {
        std::vector<int> col;
        std::vector<float> tab[2];
        if (!stg::coupling_tables(ctx->md, ctx->g.h / ctx->g.hy, ctx->g.h / ctx->g.hz, tab, &col, stg::form_of(ctx->g) != 0))
            return (int)cudaErrorInvalidValue;
        const size_t b0 = tab[0].size() * 4, b1 = tab[1].size() * 4, b2 = col.size() * 4;
        char* m = nullptr;
        cudaError_t err = cudaMalloc(&m, b0 + b1 + b2);
        if (err == cudaSuccess) err = cudaMemcpy(m, tab[0].data(), b0, cudaMemcpyHostToDevice);
        if (err == cudaSuccess) err = cudaMemcpy(m + b0, tab[1].data(), b1, cudaMemcpyHostToDevice);
        if (err == cudaSuccess) err = cudaMemcpy(m + b0 + b1, col.data(), b2, cudaMemcpyHostToDevice);
        if (err != cudaSuccess) {
            if (m) cudaFree(m);
            return (int)err;
        }
        ctx->stage_mem = m;
        ctx->stage_tab_bytes[0] = b0;
        ctx->stage_tab_bytes[1] = b1;
    }
    // last, because the active kernel may be running on the maps in place
    cudaError_t err = cudaMemcpy(ctx->stage_maps_dev, maps.data(), maps.size() * sizeof(CUtensorMap), cudaMemcpyHostToDevice);
    if (err != cudaSuccess) return (int)err;
    ctx->stage_adj_lam = ctx->stage_adj_w = nullptr;  // the adjoint's maps follow the tile
    ctx->stage_variant = (int)(v - stg::kVariants);
    ctx->tx = v->tx;
    ctx->ty = v->ty;
    ctx->tz = v->tz;
    ctx->depth = v->depth;
    ctx->tile_from_stage = true;
    return 0;
}

// the compiled (tile, depth) choices of order N, for the tuner
int stage_variants_of(int N, int precision, int* tiles, int max) {
    int n = 0;
    for (const auto& v : stg::kVariants)
        if (v.N == N && stg::fits(v, precision) && n < max) {
            tiles[4 * n] = v.tx;
            tiles[4 * n + 1] = v.ty;
            tiles[4 * n + 2] = v.tz;
            tiles[4 * n + 3] = v.depth;
            ++n;
        }
    return n;
}

// The launch fields every mode shares: geometry, the tile walk, the coupling table of a forward
// pass on class coef_cls (its sources are the other class), the status word and the wait limit.
static bool base_args(const rtpn_ctx* ctx, const stg::Variant& v, int coef_cls, stg::Args* out) {
    stg::Args a{};
    const char* m = (const char*)ctx->stage_mem;
    a.coefcol = (const float*)(coef_cls == 0 ? m : m + ctx->stage_tab_bytes[0]);
    a.colstart = (const int*)(m + ctx->stage_tab_bytes[0] + ctx->stage_tab_bytes[1]);
    a.V = ctx->g.V;
    a.nx = ctx->g.nx;
    a.ny = ctx->g.ny;
    a.nz = ctx->g.nz;
    a.bc = ctx->g.bc;
    a.inv_h = (float)(1.0 / ctx->g.h);
    a.ntx = (a.nx + v.tx - 1) / v.tx;
    a.nty = (a.ny + v.ty - 1) / v.ty;
    a.ntz = (a.nz + v.tz - 1) / v.tz;
    a.tiles = (long long)a.ntx * a.nty * a.ntz;
    // (the selection has seen to both)
    if (stages_of(v, ctx->g) >= (1ll << 31) || !stage_sized(ctx->prec, ctx->g)) return false;
    // z chunk of the tile walk: the ~one tile per SM at work at a time then spans about as many
    // tile rows in y as layers in z, across the whole x extent
    const double side = std::sqrt((double)(ctx->sms > 0 ? ctx->sms : 1) / a.ntx);
    const int kz = (int)(side + 0.5);
    a.kz = kz < 1 ? 1 : (kz > a.ntz ? a.ntz : kz);
    a.px = a.nx;
    a.sV = a.V;
    a.nc = ctx->md.nc;
    a.status = ctx->status;
    a.tickets = ctx->tickets;
    a.wait_limit = (unsigned)STAGE_WAIT_LIMIT;
    a.skip_stage = -1;
    *out = a;
    return true;
}

// a forward pass on class cls: sources through src_maps, old targets through the plane maps
// tgt_maps, new targets stored into out, whose rows are px and components sV apart (all three may be the
// context's state)
static int launch_pass(rtpn_ctx* ctx, int cls, int fac_ofs, const CUtensorMap* src_maps,
                       const CUtensorMap* tgt_maps, void* out, int px, long long sV, cudaStream_t st,
                       long long skip_stage, long long wait_limit) {
    if (ctx->stage_variant < 0) return (int)cudaErrorNotSupported;
    const stg::Variant& v = stg::kVariants[ctx->stage_variant];
    stg::Args a;
    if (!base_args(ctx, v, cls, &a)) return (int)cudaErrorInvalidValue;
    a.tgt = out;
    a.px = px;
    a.sV = sV;
    a.fac = (const float*)ctx->fac;
    a.fac_ofs = fac_ofs;
    a.maps = src_maps;
    a.tmap = tgt_maps;
    a.src_c0 = cls == 1 ? 0 : ctx->md.ne;  // the source class is the other one
    a.wait_limit = (unsigned)(wait_limit > 0xffffffffll ? 0xffffffffll : wait_limit);
    a.skip_stage = skip_stage;
    return v.launch[stg::form_of(ctx->g)](cls, ctx->prec, stg::FORWARD, a, ctx->sms, st);
}

int launch_stage(rtpn_ctx* ctx, int cls, int fac_ofs, cudaStream_t st, long long skip_stage,
                 long long wait_limit) {
    const CUtensorMap* maps = (const CUtensorMap*)ctx->stage_maps_dev;  // sources and targets: the state
    return launch_pass(ctx, cls, fac_ofs, maps, maps, ctx->u, ctx->px, ctx->sV, st, skip_stage, wait_limit);
}

int launch_stage_between(rtpn_ctx* ctx, int cls, int fac_ofs, const void* src_maps, const void* tgt_maps,
                         void* out, cudaStream_t st) {
    if (ctx->prec != RTPN_FP32) return (int)cudaErrorNotSupported;
    return launch_pass(ctx, cls, fac_ofs, (const CUtensorMap*)src_maps, (const CUtensorMap*)tgt_maps, out,
                       ctx->g.nx, ctx->g.V, st, -1, STAGE_WAIT_LIMIT);
}

size_t stage_maps_bytes(const rtpn_ctx* ctx) {
    if (ctx->stage_variant < 0) return 0;
    return (size_t)stg::MAP_KINDS * stg::nmaps_of(stg::kVariants[ctx->stage_variant], ctx->prec) *
           sizeof(CUtensorMap);
}

int stage_maps_for(rtpn_ctx* ctx, const void* state, void* maps_dev) {
    if (ctx->stage_variant < 0 || ctx->prec != RTPN_FP32 || ctx->padded()) return (int)cudaErrorNotSupported;
    const stg::Variant& v = stg::kVariants[ctx->stage_variant];
    std::vector<CUtensorMap> maps((size_t)stg::MAP_KINDS * stg::nmaps_of(v, RTPN_FP32));
    if (!stg::make_maps(maps.data(), const_cast<void*>(state), RTPN_FP32, ctx->g, ctx->g.nx, ctx->g.V, ctx->md.nc, v, stg::MAP_KINDS))
        return (int)cudaErrorInvalidValue;
    return (int)cudaMemcpy(maps_dev, maps.data(), maps.size() * sizeof(CUtensorMap), cudaMemcpyHostToDevice);
}

int launch_stage_adjoint_sources(rtpn_ctx* ctx, int tgt_cls, float* lam, const float* w, int w_planes,
                                 int fac_ofs, cudaStream_t st) {
    if (ctx->stage_variant < 0 || ctx->prec != RTPN_FP32) return (int)cudaErrorNotSupported;
    const stg::Variant& v = stg::kVariants[ctx->stage_variant];
    // tensor maps over w (every source box kind) and over lam (target planes), rebuilt when the
    // arrays change (once per adjoint call); they follow the forward maps
    const int nmap = stg::nmaps_of(v, RTPN_FP32);
    CUtensorMap* dev = (CUtensorMap*)ctx->stage_maps_dev + stg::MAP_KINDS * nmap;
    if (ctx->stage_adj_lam != lam || ctx->stage_adj_w != w) {
        std::vector<CUtensorMap> maps((size_t)(stg::MAP_KINDS + 1) * nmap);
        if (!stg::make_maps(maps.data(), const_cast<float*>(w), RTPN_FP32, ctx->g, ctx->g.nx, ctx->g.V, w_planes, v, stg::MAP_KINDS) ||
            !stg::make_maps(maps.data() + stg::MAP_KINDS * nmap, lam, RTPN_FP32, ctx->g, ctx->g.nx, ctx->g.V, ctx->md.nc, v, 1))
            return (int)cudaErrorInvalidValue;
        cudaError_t err = cudaMemcpy(dev, maps.data(), maps.size() * sizeof(CUtensorMap), cudaMemcpyHostToDevice);
        if (err != cudaSuccess) return (int)err;
        ctx->stage_adj_lam = lam;
        ctx->stage_adj_w = w;
    }
    // the coupling table of a forward pass on the target class: its sources are the other class
    stg::Args a;
    if (!base_args(ctx, v, tgt_cls, &a)) return (int)cudaErrorInvalidValue;
    a.tgt = lam;
    a.fac = fac_ofs >= 0 ? (const float*)ctx->fac : nullptr;  // lam_B <- alpha_B lam_B folded in
    a.fac_ofs = fac_ofs >= 0 ? fac_ofs : 0;
    a.maps = dev;
    a.tmap = dev + stg::MAP_KINDS * nmap;
    a.src_c0 = 0;  // w holds only the source class, in its local order
    a.nc = w_planes;
    return v.launch[stg::form_of(ctx->g)](tgt_cls, RTPN_FP32, stg::ADJ_SOURCES, a, ctx->sms, st);
}

}  // namespace rtpn
