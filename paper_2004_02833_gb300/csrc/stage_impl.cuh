// TMA-staged substep kernel with a compact column loop (FP32 arithmetic, FP32 or BF16 storage).
//
// Arithmetic as in the register-window kernel (window_impl.cuh): the frozen class is swept column by
// column in |m|; every source value yields three half-grid differences (Section 2.1) that are
// scattered into the accumulators of its <= 10 targets (Eqs. 4-5; Section 3.2's unrolled sparse
// product), and a target column is finished, by Eq. (5), once the next source column is in.  What
// differs:
//
//  * A thread advances both types (cos / sin) of one cell, a type per lane of packed FP32 pairs:
//    targets of type T take their z and x differences from sources of type T and their y differences
//    from sources of the other type (Eq. 3's Mx and Mz keep the type, My swaps it), so the two lanes
//    run the same code and share one coupling constant for x and y.  Each thread keeps three columns
//    of N/2 + 1 accumulator pairs.  (Two threads per cell, one per type, took twice the instructions
//    for the same cells: P39 160^3 FP32, 11.0 ms a pass against 7.1 ms now.)
//  * The column sweep is a runtime loop whose body handles one column for every l slot; the three
//    live target columns are register arrays that change roles from column to column (the loop is
//    unrolled by three), so the body is the same for every column and fits the instruction cache.
//  * A column is moved in NCH sub-stages of K = 4 or 5 slots, so that a stage buffer is small and the
//    tile can be wide (up to 96 cells): TMA rows of 256 to 384 bytes and up to 12 consumer warps for the
//    same shared memory.  A target slot is finished in the sub-stage that brings its last source.
//  * Two producer warps, one per type, move each sub-stage into shared memory with the Tensor Memory
//    Accelerator (cp.async.bulk.tensor): one box per box kind holding all its components of the
//    (type, |m|) run at once (a tensor map per box length).  Every box kind has the same volume per
//    component, U = TY * TX elements: the tile as TZ plane boxes [E][1][TY][TX], the y halo row
//    [E][TZ][1][TX], the z halo plane [E][1][TY][TX] and the x halo [E][TZ][RY][XW] (XW * RY = TX: an
//    aligned group of XW columns around the neighbour the partners read, with RY >= TY rows).  So
//    slot k of every region sits at k * U elements and each thread reaches all its operands through a
//    few base addresses fixed once per column plus compile-time offsets: no address arithmetic per
//    slot.  Periodic halos use wrapped coordinates; vacuum halos use out-of-range coordinates, which
//    the TMA unit fills with zeros.  The same stage carries the tile boxes of the target slots it
//    finishes and the coupling constants (a plain bulk copy).  The issue of the boxes bounds the
//    copies (about 100 cycles a box from one warp, copies alone): P39 160^3, 7.2 ms with one producer
//    warp, 5.5 ms with two, 4.4 ms with everything but the issue itself computed by the whole warp
//    (uniform registers) instead of by one lane.  NB stage buffers form a ring with a full / empty
//    mbarrier pair each, so up to NB - 1 stages are in flight while one is computed.
//
// What bounds it (GB300, FP32, a pass, before -> now, of the 6697 GB/s copy): P39 160^3 11.0 -> 7.1 ms
// (5.6 TB/s, 83 %): the latency of a warp's own instructions, 10 consumer warps with 168 registers (120
// accumulators); P19 96 x 96 x 128 0.54 ms (5.2 TB/s); P15 96^3 0.41 -> 0.27 ms (5.1 TB/s, 77 %); P7 128^3
// 0.46 -> 0.19 ms (4.3 TB/s): barriers and copies per stage.
//
// CTAs are persistent (one or two per SM) and take tiles by ticket (an atomic counter) in z-chunked order (z
// fastest inside a chunk of kz tile layers, then x, then y), so the CTAs at work at any time cover a compact
// block and read one another's halos from L2.  With fixed shares instead, a pass waited for the CTAs that
// started late because another stream's kernel held their SMs (three P39 160^3 contexts in turn, two
// steps and the state out each: 54.2 ms against 42.4 with tickets; one pass alone 7.4 -> 7.1 ms).
// Every mbarrier wait is bounded: one that runs out sets a status bit;
// a consumer then neither waits nor hands a buffer back for the rest of its tile (whose results are
// undefined, as the caller is told), so that the producers run out of buffers instead of reusing one
// whose copies are in flight; a producer leaves after a bounded wait for the copies it issued.
#pragma once

#include <cuda.h>

#include "window_impl.cuh"

namespace rtpn {
namespace stg {

using win::class_size;
using win::column_len;
using win::first_l;
using win::ntypes;
using win::static_for;

constexpr int kMaxSlots = 24;  // tensor maps of a kind, at most
// The slots of a sub-stage run in blocks of straight-line code, skipped where the column starts
// above them; slots of a block below the first source carry zero constants and read finite shared
// memory.
constexpr int kBlock = 2;
// A sub-stage's last block takes the remainder, so a block has up to 2 kBlock - 1 slots; one that holds the
// column's first source may start that many less one below it.
constexpr int kBelow = 2 * kBlock - 2;
// Producer warps: one for each type's boxes of every stage.
constexpr int kProducers = 2;

constexpr unsigned STATUS_TIMEOUT = 1u;
constexpr unsigned STATUS_CHECK = 2u;  // a self-check failed (builds with RTPN_STAGE_CHECKS)
// Coupling constants per source slot (l, M): six (cos, sin) pairs, one lane per target type T: z to l-1,
// z to l+1 (target column M), x and y to column M+1 (l-1, l+1), and, negated, to column M-1 (l-1, l+1).
// Mx and My couple (l, M) to (l +- 1, M +- 1) with entries of the same magnitude (both come from
// Omega_x +- i Omega_y), and the sign of the y entry against the x entry depends on (T, parity of M,
// side) only: + into column M+1 for T = 0 and even M, and the other sign for each of T = 1, odd M and
// column M-1.  So one constant serves both axes: with dx the x difference of the own type's source and
// dy the y difference of the other type's, a target takes k dx + k (s dy) from column M-1 and
// (-k)(-dx) + (-k)(s dy) from column M+1, s = +-1 the same for the whole column.
constexpr int CPAD = 6;       // constants per slot and type
constexpr int KPAIRS = CPAD;  // pairs per slot
// Cells with h_y != h_x (form SC): the y constants carry h / h_y, rounded once from the product, so they are
// no longer the x ones: four more pairs per slot, to column M+1 and M-1 (l-1, l+1 each).  (Scaling the
// differences by an FP32 h / h_y instead rounds twice, with one error for all of them: 8 to 10 % more
// error at h / h_y = 1/1.1, 0.6 and 1/1.7 after forty P15 passes.)
template <bool SC>
RTPN_HD constexpr int slot_pairs() {
    return SC ? 10 : KPAIRS;
}

// What a pass computes.  FORWARD: targets u_A' = alpha u_A - beta acc (Eq. 5; the u_0 factors for
// l = 0).  ADJ_SOURCES: the transpose of a substep's coupling for the dual multipliers,
// lam_B' = alpha_B lam_B + acc / h with the sources the weights w_A = beta_A lam_A of the substep on
// class A (same stencil rule and coefficient table as a forward pass on class B: see
// csrc/adjoint.cu); alpha_B, when factors are given, is the factor of the later substep on class B
// whose pull-back lam_B <- alpha_B lam_B is folded in here.
constexpr int FORWARD = 0, ADJ_SOURCES = 1;

// Tensor maps of one array: kind k in {MAP_PLANE, MAP_YROW, MAP_XGRP} for every box length
// E = 1, 2, ..., NMAP (index k * nmaps + E - 1).
constexpr int MAP_PLANE = 0;  // [E][1][TY][TX]: a tile plane or the z halo plane (also target boxes)
constexpr int MAP_YROW = 1;   // [E][TZ][1][TX]: the y halo row
constexpr int MAP_XGRP = 2;   // [E][TZ][RY][XW]: the x halo group
constexpr int MAP_KINDS = 3;

struct Args {
    void* tgt;              // target array written (u for a forward pass, lam for ADJ_SOURCES)
    const float* fac;
    const float* coefcol;   // [column 0..N][type][slot q 0..N/2][CPAD] of the source class (0 for l < M)
    const int* colstart;    // [2][N+2]: first local index of column M in class 0 / class 1
    long long V;            // cells: stride of the factor planes (dense rows)
    int nx, ny, nz, bc;
    int fac_ofs;
    float inv_h;
    int ntx, nty, ntz;
    int kz;                 // tile layers per z chunk of the walk
    long long tiles;
    const CUtensorMap* maps;  // MAP_KINDS * nmaps tensor maps over the source array
    const CUtensorMap* tmap;  // nmaps MAP_PLANE maps over the target array
    int src_c0;               // first component of the source class in the source array
    int nc;                   // components (bound of the 4th tensor coordinate)
    unsigned* status;       // device status word (STATUS_TIMEOUT on a wait that ran out)
    unsigned wait_limit;    // try_wait polls (each up to WAIT_HINT_NS) before giving up
    unsigned* tickets;      // [0] tiles handed out past the first round, [1] CTAs that are done (both 0 between passes)
    long long skip_stage;   // stage index never issued (a wait that must run out); -1 normally
    int px = 0;             // row pitch of the target array and stride of its components
    long long sV = 0;
    // Scale of the y differences: 1, other than in a host run without form SC.  An argument and no constant, because with
    // the constant the compiler spills: P39 200^3 FP32, odd pass 15.2 ms against 14.7.
    float sy = 1.f;
};

__host__ __device__ constexpr int pad128(int bytes) { return (bytes + 127) / 128 * 128; }

// Tile indices handed from the producer that draws them to the other warps of the CTA.
constexpr int kNextRing = 4;

// Width XW of the x halo box: the widest group of 16-byte aligned columns that divides TX and
// leaves RY = TX / XW >= TY rows (so the box volume per component is TZ * TX = U when TY == TZ).
__host__ __device__ constexpr int xhalo_width(int tx, int ty, int es) {
    int best = 0;
    for (int w = 16 / es; w <= tx; w += 16 / es)
        if (tx % w == 0 && tx / w >= ty) best = w;
    return best;
}

// NCH: sub-stages of a column (each K = ceil((N/2 + 1) / NCH) source slots).  SC: with y constants of their own.
template <int N, int A, typename S, int TX, int TY, int TZ, int NB, int NCH = 1, bool SC = false>
struct Layout {
    static constexpr int B = 1 - A;
    static constexpr int ES = (int)sizeof(S);
    static constexpr int G = 16 / ES;                 // elements of an aligned 16-byte group
    static constexpr int NLC = N / 2 + 1;             // slots of the longest run
    static constexpr int K = (NLC + NCH - 1) / NCH;   // source slots of a sub-stage
    static constexpr int KT = NCH == 1 ? K : K + 1;   // target slots of a sub-stage, at most
    static constexpr int NL = KT;                     // longest box
    static constexpr int NMAP = KT;                   // box lengths (tensor maps) per kind
    static constexpr int U = TY * TX;                 // elements of one component in every box
    static constexpr int UB = U * ES;
    static constexpr int XW = xhalo_width(TX, TY, ES);
    static constexpr int RY = XW > 0 ? TX / XW : 1;
    static constexpr int CELLS = TX * TY * TZ;
    static constexpr int CONSUMER_WARPS = CELLS / 32;
    static constexpr int THREADS = CELLS + 32 * kProducers;  // one thread per cell + the producers
    static constexpr int REG = pad128(K * UB);        // one source region: K components of one box kind
    static constexpr int REGT = pad128(KT * UB);      // one target region
    // regions of one type's sources: TZ tile planes, then the y halo, z halo and x halo
    static constexpr int KY = TZ, KZ = TZ + 1, KX = TZ + 2, NKIND = TZ + 3;
    static constexpr int SRC_T = NKIND * REG;
    static constexpr int TGT_T = TZ * REGT;           // tile planes of one type's targets
    static constexpr int PAIRS = slot_pairs<SC>();      // pairs of constants per slot
    static constexpr int COEF_COL = 2 * K * PAIRS * 4;  // a sub-stage's coupling constants
    // buffer layout: target planes, type-0 sources, type-1 sources, coupling constants.  A block of
    // the sweep may read up to kBelow slots below a source region; with the targets first, such reads
    // stay on state data (or the zeros the ring starts with) in the same buffer, never on the
    // coupling constants, whose bits need not be finite in the storage type.
    static constexpr int TGTO = 0;
    static constexpr int SRCO = 2 * TGT_T;
    static constexpr int COEFO = SRCO + 2 * SRC_T;
    static constexpr int BUF = COEFO + pad128(COEF_COL);  // one stage buffer
    static constexpr int BARS = pad128(2 * NB * 8);
    static constexpr int NEXT = 128;                      // the next tiles' indices (kNextRing)
    static constexpr int BYTES = NB * BUF + BARS + NEXT + 128;  // ring, mbarriers, tiles, alignment slack
    static_assert(TY == TZ, "every box kind has the volume TY * TX per component only if TY == TZ");
    static_assert(TX % G == 0, "tile width must be a multiple of the 16-byte group");
    static_assert(CELLS % 32 == 0, "the tile's cells must fill whole warps");
    static_assert(NB >= 2 && NB <= 8, "two to eight stage buffers");
    static_assert(2 * TGT_T >= kBelow * UB && REG >= kBelow * UB, "a block's reads below a region stay in the one before");
    static_assert(NCH == 1 || K >= 2, "a sub-stage of class 1 finishes one slot behind its sources");
    // the ring fits 227 KB of shared memory per CTA, and an x halo group exists for this element
    // size (a tile too narrow for RY >= TY rows of 16-byte groups is compiled for FP32 only)
    static constexpr bool FITS = BYTES <= 232448 && XW > 0;
};

// First slot of source column i (class B), and the sub-stage a column starts with.
template <int N, int A>
RTPN_HD constexpr int first_source(int i) {
    return (int)(((unsigned)i + (((unsigned)i ^ (unsigned)(1 - A)) & 1u)) >> 1);  // first_l(i, B) / 2
}
template <int N, int A, int NCH>
RTPN_HD constexpr int first_chunk(int i) {
    constexpr int K = (N / 2 + 1 + NCH - 1) / NCH;
    const int c = first_source<N, A>(i) / K;
    return c < NCH - 1 ? c : NCH - 1;
}
// sub-stages of one tile
template <int N, int A, int NCH>
RTPN_HD constexpr int tile_stages() {
    int n = 0;
    for (int i = 0; i < N + 2; ++i) n += NCH - first_chunk<N, A, NCH>(i);
    return n;
}
// Target slots [lo, hi) of column i - 1 that are complete after sub-stage C of source column i: a
// source l reaches l +- 1, so class 0 (even l) is complete up to the same slot, class 1 up to the one
// before, and the last sub-stage completes the rest.
template <int N, int A, int NCH>
RTPN_HD constexpr int window_lo(int C) {
    constexpr int K = (N / 2 + 1 + NCH - 1) / NCH;
    return C == 0 ? 0 : C * K - A;
}
template <int N, int A, int NCH>
RTPN_HD constexpr int window_hi(int C) {
    constexpr int K = (N / 2 + 1 + NCH - 1) / NCH;
    constexpr int NLA = (N - A) / 2 + 1;
    const int h = C * K + K - A;
    return C == NCH - 1 || h > NLA ? NLA : h;
}

// Sign of the y against the x coupling into column M+1 for target type T.
RTPN_HD constexpr float y_sign(int M, int T) { return ((M ^ T) & 1) ? -1.f : 1.f; }

// The coupling constants of the staged kernel (host; the library and its host check program):
// per target class A, the constants of the source class by column and slot q
// ([N+1][N/2+1][KPAIRS][2], layout above; slots of l < M stay zero), from the model's coupling
// (win::coef_table).  The kernel applies 1/h of x; the z constants carry
// sz = h / h_z (exactly 1 for cubic cells); scaled: the layout of form SC, whose y constants carry sy = h / h_y.  col: the first local index of column M in
// class P at col[P (N + 2) + M].  False if the model's x and y couplings do not share their magnitudes
// and signs as above.
inline bool coupling_tables(const Model& md, double sy, double sz, std::vector<float> tab[2], std::vector<int>* col,
                            bool scaled = false) {
    const int N = md.N, nl = N / 2 + 1, pairs = scaled ? slot_pairs<true>() : slot_pairs<false>();
    col->assign(2 * (N + 2), 0);
    for (int P = 0; P < 2; ++P) {
        int acc = 0;
        for (int M = 0; M <= N + 1; ++M) {
            (*col)[P * (N + 2) + M] = acc;
            if (M <= N) acc += ntypes(M) * column_len(N, M, P);
        }
    }
    for (int A = 0; A < 2; ++A) {
        const int B = 1 - A;
        std::vector<float> t10;  // [local source index of class B][10]
        if (!win::coef_table(md, A, &t10)) return false;
        tab[A].assign((size_t)(N + 1) * nl * 2 * pairs, 0.f);
        for (int M = 0; M <= N; ++M)
            for (int j = 0; j < column_len(N, M, B); ++j) {
                const int q = first_l(M, B) / 2 + j;  // the source's slot (l - B) / 2
                float* d = &tab[A][((size_t)M * nl + q) * pairs * 2];
                // relations of the source of type t (null if the type is absent)
                auto rel = [&](int t) {
                    const int len = column_len(N, M, B);
                    return t < ntypes(M) ? &t10[(size_t)((*col)[B * (N + 2) + M] + t * len + j) * 10] : nullptr;
                };
                for (int T = 0; T < 2; ++T) {
                    const float *own = rel(T), *oth = rel(1 - T);
                    for (int r = 0; r < 2 && own; ++r) d[r * 2 + T] = (float)(own[r] * sz);
                    for (int side = 0; side < 2; ++side)  // column M+1, column M-1
                        for (int dl = 0; dl < 2; ++dl) {
                            const float x = own ? own[(side == 0 ? 4 : 2) + dl] : 0.f;
                            const float y = oth ? oth[(side == 0 ? 8 : 6) + dl] : 0.f;
                            const float s = side == 0 ? y_sign(M, T) : -y_sign(M, T);
                            // at |m| = 0 only one of the two sources exists
                            if (M > 0 ? y != s * x : (x != 0.f && y != 0.f)) return false;
                            const float k = own ? x : scaled ? 0.f : s * y;
                            d[(2 + 2 * side + dl) * 2 + T] = side == 0 ? k : -k;
                            if (scaled) d[(6 + 2 * side + dl) * 2 + T] = (float)(y * sy) * y_sign(M, T);
                        }
                }
            }
    }
    return true;
}

// ---------------------------------------------------------------- PTX helpers
__device__ __forceinline__ unsigned smem_addr(const void* p) {
    return static_cast<unsigned>(__cvta_generic_to_shared(p));
}
__device__ __forceinline__ void mbar_init(unsigned bar, unsigned count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(unsigned bar, unsigned bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes)
                 : "memory");
}
__device__ __forceinline__ void mbar_arrive(unsigned bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
// One poll: the thread may sleep up to WAIT_HINT_NS for the phase to complete (it wakes when it
// does), so a warp that waits for its data spends few issue slots on the poll loop.
constexpr unsigned WAIT_HINT_NS = 2000;
__device__ __forceinline__ bool mbar_try_wait(unsigned bar, unsigned parity) {
    unsigned ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(bar), "r"(parity), "n"(WAIT_HINT_NS)
        : "memory");
    return ok != 0;
}
__device__ __forceinline__ void tma_load_4d(unsigned dst, const CUtensorMap* map, int x, int y, int z,
                                            int c, unsigned bar) {
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes"
        " [%0], [%1, {%2, %3, %4, %5}], [%6];" ::"r"(dst),
        "l"(reinterpret_cast<unsigned long long>(map)), "r"(x), "r"(y), "r"(z), "r"(c), "r"(bar)
        : "memory");
}
__device__ __forceinline__ void bulk_load(unsigned dst, const void* src, unsigned bytes, unsigned bar) {
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
        "l"(reinterpret_cast<unsigned long long>(src)), "r"(bytes), "r"(bar)
        : "memory");
}
// true on one lane of the (converged) warp
__device__ __forceinline__ bool elect_one() {
    unsigned p;
    asm volatile("{\n\t.reg .pred q;\n\telect.sync _|q, 0xffffffff;\n\tselp.u32 %0, 1, 0, q;\n\t}" : "=r"(p));
    return p != 0;
}
// bounded wait of a whole warp on one mbarrier phase; false if it ran out (the same for every lane)
__device__ __forceinline__ bool wait_phase(unsigned bar, unsigned parity, unsigned limit) {
    for (unsigned i = 0; i < limit; ++i)
        if (__all_sync(0xffffffffu, mbar_try_wait(bar, parity))) return true;
    return false;
}

// a stored value at base + byte_off of a stage buffer, as FP32 (host and device: the host check
// program runs the consumers' column work over a bounds-checked copy of the buffer)
template <typename S>
RTPN_HD float lds(const unsigned char* base, int byte_off) {
    RTPN_CHECK_PTR(base + byte_off);
    if constexpr (sizeof(S) == 4) {
        return *reinterpret_cast<const float*>(base + byte_off);
    } else {
        return __bfloat162float(*reinterpret_cast<const __nv_bfloat16*>(base + byte_off));
    }
}

// Optional self-checks (compile with -DRTPN_STAGE_CHECKS): an index that breaks the layout sets
// STATUS_CHECK and the access is skipped.  status[1] holds the id of the first failed check,
// status[2] a value of it, status[7] the block.
#ifdef RTPN_STAGE_CHECKS
__device__ __forceinline__ bool scheck_fail(unsigned* st, unsigned id, unsigned val, unsigned aux) {
    atomicOr(st, STATUS_CHECK);
    if (atomicCAS(st + 1, 0u, id) == 0u) {
        st[2] = val;
        st[7] = aux;
    }
    return false;
}
#define RTPN_SCHECK_ID(cond, id, val) ((cond) ? true : scheck_fail(a.status, (id), (unsigned)(val), blockIdx.x))
#else
#define RTPN_SCHECK_ID(cond, id, val) true
#endif
#define RTPN_SCHECK(cond) RTPN_SCHECK_ID(cond, __LINE__, 0)

// Tile geometry: origin, valid extents, halo coordinates ([axis][side], side 1 = upper) and, per
// side, the origin of the x halo group box and the element of the neighbour column inside it.
struct TileGeo {
    int x0, y0, z0, wx, wy, wz;
    int hc[3][2];
    int hx_start[2], hx_elem[2];
};

// tile t of the walk: chunks of kz z-layers; inside a chunk z fastest, then x, then y
__host__ __device__ __forceinline__ void tile_coords(unsigned t, int ntx, int nty, int ntz, int kzc, int* bx,
                                                     int* by, int* bz) {
    const unsigned per_chunk = (unsigned)kzc * ntx * nty;
    const unsigned full = (unsigned)(ntz / kzc);
    unsigned chunk, r, kz;
    if (t < full * per_chunk) {
        chunk = t / per_chunk;
        r = t - chunk * per_chunk;
        kz = kzc;
    } else {
        chunk = full;
        r = t - full * per_chunk;
        kz = ntz - full * kzc;
    }
    *bz = (int)(chunk * kzc + r % kz);
    const unsigned rest = r / kz;
    *bx = (int)(rest % ntx);
    *by = (int)(rest / ntx);
}

// G: elements of a 16-byte group (the x halo box starts on one)
template <int TX, int TY, int TZ, int G>
__host__ __device__ __forceinline__ TileGeo tile_geo(const Args& a, unsigned t) {
    TileGeo g;
    int bx, by, bz;
    tile_coords(t, a.ntx, a.nty, a.ntz, a.kz, &bx, &by, &bz);
    g.x0 = bx * TX;
    g.y0 = by * TY;
    g.z0 = bz * TZ;
    g.wx = min(TX, a.nx - g.x0);
    g.wy = min(TY, a.ny - g.y0);
    g.wz = min(TZ, a.nz - g.z0);
    const bool periodic = a.bc == RTPN_BC_PERIODIC;
    const int o[3] = {g.x0, g.y0, g.z0}, w[3] = {g.wx, g.wy, g.wz}, n[3] = {a.nx, a.ny, a.nz};
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        int up = o[d] + w[d], lo = o[d] - 1;
        if (periodic) {
            if (up >= n[d]) up -= n[d];
            if (lo < 0) lo += n[d];
        }
        g.hc[d][1] = up;
        g.hc[d][0] = lo;
    }
    // the neighbour column xn sits at element xn - start of a box that starts on the group holding it
#pragma unroll
    for (int s = 0; s < 2; ++s) {
        const int xn = g.hc[0][s];
        const int st = xn >= 0 ? (xn / G) * G : -G;
        g.hx_start[s] = st;
        g.hx_elem[s] = xn - st;
    }
    return g;
}

// Source x slot: 1 (read at i+1 by its partners) iff (M even) == (cos type); z slot: 1 iff l+M even.
__host__ __device__ __forceinline__ int dir_x(int M, int t) { return ((M & 1) == 0) == (t == 0) ? 1 : -1; }

// ---------------------------------------------------------------- the stage plan
// One TMA box of a stage: which tensor map (array, kind, box length), its start coordinates and
// where it lands in the stage buffer.  Host and device: the producer issues it, the host check
// program copies it.
struct BoxJob {
    int valid;    // 0: this box is not part of the stage
    int target;   // 1: a plane box of the target array (map a.tmap + emap), 0: of the source array
    int kind;     // MAP_PLANE, MAP_YROW or MAP_XGRP (source array)
    int emap;     // box length index: E = emap + 1 components
    int x, y, z, c;
    int dst;      // byte offset of the box in the stage buffer
};

// The runs of sub-stage C of stage i, the same for every box: slots of source column i of class B and of
// target column i - 1 of class A (box lengths, types present), the full runs and where in them the
// boxes start, and the slots the boxes start with.
struct StageRuns {
    int len, nt, lenA, ntA;
    int run, ofs, runA, ofsA;
    int q, qA;
};
template <int N, int A, int NCH = 1>
RTPN_HD StageRuns stage_runs(int i, int C = 0) {
    constexpr int B = 1 - A;
    constexpr int K = (N / 2 + 1 + NCH - 1) / NCH;
    constexpr int NLB = (N - B) / 2 + 1;
    StageRuns r;
    r.run = column_len(N, i, B);  // none at i = N + 1
    const int fq = first_source<N, A>(i);
    r.q = fq > C * K ? fq : C * K;
    const int e = C * K + K < NLB ? C * K + K : NLB;
    r.len = i <= N && e > r.q ? e - r.q : 0;
    r.ofs = r.q - fq;
    r.nt = r.len > 0 ? ntypes(i) : 0;
    r.runA = i >= 1 ? column_len(N, i - 1, A) : 0;
    const int q0 = i >= 1 ? first_l(i - 1, A) / 2 : 0, lo = window_lo<N, A, NCH>(C), hi = window_hi<N, A, NCH>(C);
    r.qA = q0 > lo ? q0 : lo;
    r.lenA = i >= 1 && hi > r.qA ? hi - r.qA : 0;
    r.ofsA = r.qA - q0;
    r.ntA = r.lenA > 0 ? ntypes(i - 1) : 0;
    return r;
}

// Source box K of type t of a sub-stage of stage i (runs r) of the tile with geometry g: K = 0 .. TZ - 1 the
// tile planes, then the y halo row, the z halo plane, the x halo group; offB is the first local index of
// source column i in class B.
template <int N, int A, typename S, int TX, int TY, int TZ, int NB, int NCH, int K>
RTPN_HD BoxJob source_box(const Args& a, const TileGeo& g, int i, const StageRuns& r, int offB, int t) {
    using L = Layout<N, A, S, TX, TY, TZ, NB, NCH>;
    constexpr int B = 1 - A;
    BoxJob bj;
    bj.valid = t < r.nt;
    bj.target = 0;
    bj.emap = r.len - 1;
    bj.c = a.src_c0 + offB + t * r.run + r.ofs;  // first component of the box
    bj.dst = L::SRCO + t * L::SRC_T + K * L::REG;
    bj.x = g.x0;
    bj.y = g.y0;
    bj.z = g.z0;
    bj.kind = MAP_PLANE;
    if constexpr (K < TZ) {             // tile plane z0 + K
        bj.z = g.z0 + K;
    } else if constexpr (K == L::KY) {  // cos-type sources are read at y+1, sin-type at y-1
        bj.kind = MAP_YROW;
        bj.y = t == 0 ? g.hc[1][1] : g.hc[1][0];
    } else if constexpr (K == L::KZ) {  // z slot 1 (l + M even) is read at z+1
        bj.z = ((B + i) & 1) == 0 ? g.hc[2][1] : g.hc[2][0];
    } else {                            // x slot 1 is read at x+1 (upper halo group)
        bj.kind = MAP_XGRP;
        bj.x = dir_x(i, t) > 0 ? g.hx_start[1] : g.hx_start[0];
    }
    return bj;
}
// Target plane lz of type t; offA is the first local index of target column i - 1 in class A.
template <int N, int A, typename S, int TX, int TY, int TZ, int NB, int NCH>
RTPN_HD BoxJob target_box(const TileGeo& g, const StageRuns& r, int offA, int t, int lz) {
    using L = Layout<N, A, S, TX, TY, TZ, NB, NCH>;
    BoxJob bj;
    bj.valid = t < r.ntA;
    bj.target = 1;
    bj.kind = MAP_PLANE;
    bj.emap = r.lenA - 1;
    bj.x = g.x0;
    bj.y = g.y0;
    bj.z = g.z0 + lz;
    bj.c = (A == 0 ? 0 : class_size(N, 0)) + offA + t * r.runA + r.ofsA;
    bj.dst = L::TGTO + t * L::TGT_T + lz * L::REGT;
    return bj;
}

// Box j of the plan: 0 .. 2 NKIND - 1 the source boxes (type j / NKIND, kind j % NKIND), then the target
// planes (type, plane).
template <int N, int A, typename S, int TX, int TY, int TZ, int NB, int NCH>
RTPN_HD BoxJob stage_box(const Args& a, const TileGeo& g, int i, const StageRuns& r, int offA, int offB, int j) {
    using L = Layout<N, A, S, TX, TY, TZ, NB, NCH>;
    constexpr int NK = L::NKIND;
    BoxJob bj{0, 0, 0, 0, 0, 0, 0, 0, 0};
    if (j >= 2 * NK)
        return j < 2 * NK + 2 * TZ ? target_box<N, A, S, TX, TY, TZ, NB, NCH>(g, r, offA, (j - 2 * NK) / TZ, (j - 2 * NK) % TZ)
                                   : bj;
    static_for<NK>([&](auto kk) {
        constexpr int K = decltype(kk)::value;
        if (j % NK == K) bj = source_box<N, A, S, TX, TY, TZ, NB, NCH, K>(a, g, i, r, offB, j / NK);
    });
    return bj;
}

// coupling-constant slots of sub-stage C that exist
template <int N, int NCH>
RTPN_HD constexpr int coef_slots(int C) {
    constexpr int NLC = N / 2 + 1, K = (NLC + NCH - 1) / NCH;
    return C * K + K <= NLC ? K : NLC - C * K;
}
// bytes that type t's boxes of a sub-stage with runs r bring into the buffer (the coupling constants
// come with type 0), and those of both types
template <int N, int A, typename S, int TX, int TY, int TZ, int NB, int NCH, bool SC = false>
RTPN_HD unsigned type_bytes(const StageRuns& r, int C, int t) {
    using L = Layout<N, A, S, TX, TY, TZ, NB, NCH, SC>;
    return (unsigned)(((t < r.nt ? L::NKIND * r.len : 0) + (t < r.ntA ? TZ * r.lenA : 0)) * L::UB) +
           (t == 0 && r.nt > 0 ? (unsigned)coef_slots<N, NCH>(C) * (2 * L::PAIRS * 4) : 0u);
}
template <int N, int A, typename S, int TX, int TY, int TZ, int NB, int NCH>
RTPN_HD unsigned stage_bytes(const StageRuns& r, int C = 0) {
    return type_bytes<N, A, S, TX, TY, TZ, NB, NCH>(r, C, 0) + type_bytes<N, A, S, TX, TY, TZ, NB, NCH>(r, C, 1);
}

// What the ring rests on when a wait runs out (also run by a host model of its barriers).  Stage s uses
// buffer s % nb; phase s / nb of the buffer's full barrier is the one its copies complete.
// A consumer warp whose wait ran out (its limit is then 0) hands no buffer back: the buffer may have copies in
// flight, or none issued, and a producer given it would arrive on a phase that is not complete.
RTPN_HD constexpr bool hands_back(unsigned limit) { return limit != 0; }
// A producer that issued the stages below s waits for those from here on before its CTA ends: the earlier
// ones were handed back.
RTPN_HD constexpr int drain_first(int s, int nb) { return s > nb ? s - nb : 0; }
RTPN_HD constexpr unsigned full_parity(int s, int nb) { return (unsigned)(s / nb) & 1u; }

// Producer warp t: issues the copies of type t (and for t = 0 the coupling constants) of every sub-stage
// of this CTA's sequence into the ring.  One lane issues; everything else is the same for the warp.
template <int N, int A, typename S, int TX, int TY, int TZ, int NB, int NCH, bool SC>
__device__ __forceinline__ void stage_producer(const Args& a, unsigned char* bufs, unsigned full0,
                                               unsigned empty0, volatile unsigned* next, int t) {
    using L = Layout<N, A, S, TX, TY, TZ, NB, NCH, SC>;
    constexpr int B = 1 - A;
    constexpr int NST = N + 2;
    const int lane = threadIdx.x & 31;
    const CUtensorMap* maps = a.maps;
    // first local index of source column i in class B and of target column i - 1 in class A,
    // advanced column by column (no table loads on the producer's path)
    int offB = 0, offA = 0;
    // the maps were written by the host before the launch; make them visible to the async proxy
    for (int k = 0; k < MAP_KINDS * L::NMAP; ++k)
        asm volatile("fence.proxy.tensormap::generic.acquire.gpu [%0], 128;" ::"l"(maps + k) : "memory");
    for (int k = 0; k < L::NMAP; ++k)
        asm volatile("fence.proxy.tensormap::generic.acquire.gpu [%0], 128;" ::"l"(a.tmap + k) : "memory");

    constexpr int TS = tile_stages<N, A, NCH>();
    static_assert(TS >= NB + 2, "a tile's second stage is consumed before the next tile is issued");
    int s = 0;
    bool failed = false;
    int b = 0;
    unsigned ph = 0;  // phase parity of buffer b's current use (flips when b wraps)
    unsigned tile = blockIdx.x, ticket = 0;
    for (unsigned k = 0;; ++k) {
      TileGeo g{};
      int i = 0, C = first_chunk<N, A, NCH>(0);
      int j = 0;
      for (; j < TS; ++j, ++s) {
        const unsigned full = full0 + 8 * b;
        if (s >= NB && !wait_phase(empty0 + 8 * b, ph ^ 1u, a.wait_limit)) {
            failed = true;  // the consumers did not release the buffer's previous stage
            break;
        }
        // The next tile: producer 0 draws it while the tile's first stage is issued and hands it on before
        // the arrival of the second; the consumers have it with that stage, producer 1 with their release.
        if (j == 0) {
            if (k > 0) tile = next[k % kNextRing];
            if (tile >= (unsigned long long)a.tiles) break;
            g = tile_geo<TX, TY, TZ, L::G>(a, tile);
            offA = offB = 0;
            if (t == 0 && lane == 0) ticket = atomicAdd(a.tickets, 1u);
        } else if (j == 1 && t == 0) {
            if (lane == 0) next[(k + 1) % kNextRing] = gridDim.x + ticket;
            __syncwarp();
        }
        const unsigned buf = smem_addr(bufs + b * L::BUF);
        const StageRuns r = stage_runs<N, A, NCH>(i, C);
        const unsigned bytes = type_bytes<N, A, S, TX, TY, TZ, NB, NCH, SC>(r, C, t);
        auto issue = [&](const BoxJob& bj) {
            // sources: components of the source array (a.nc); targets: of a full state array (u or lam)
            const int cmax = bj.target ? class_size(N, 0) + class_size(N, 1) : a.nc;
            if (RTPN_SCHECK_ID(bj.c >= 0 && bj.c < cmax && bj.emap < L::NMAP, 101, bj.c)) {
                const CUtensorMap* mp = bj.target ? a.tmap + bj.emap : maps + bj.kind * L::NMAP + bj.emap;
                tma_load_4d(buf + bj.dst, mp, bj.x, bj.y, bj.z, bj.c, full);
            }
        };
        if (s != a.skip_stage) {
            if (elect_one()) {
                mbar_expect_tx(full, bytes);
                if (t < r.nt) {
                    static_for<L::NKIND>([&](auto kk) {
                        issue(source_box<N, A, S, TX, TY, TZ, NB, NCH, decltype(kk)::value>(a, g, i, r, offB, t));
                    });
                    if (t == 0)
                        bulk_load(buf + L::COEFO, a.coefcol + (long long)(i * L::NLC + C * L::K) * (2 * L::PAIRS),
                                  coef_slots<N, NCH>(C) * (2 * L::PAIRS * 4), full);
                }
                if (t < r.ntA)
                    static_for<TZ>([&](auto zz) {
                        issue(target_box<N, A, S, TX, TY, TZ, NB, NCH>(g, r, offA, t, decltype(zz)::value));
                    });
            }
            __syncwarp();
        }
        if (++b == NB) {
            b = 0;
            ph ^= 1u;
        }
        // the next sub-stage: of this column or the next
        if (++C == NCH) {
            offB += ntypes(i) * column_len(N, i, B);
            if (i >= 1) offA += ntypes(i - 1) * column_len(N, i - 1, A);
            if (++i < NST) C = first_chunk<N, A, NCH>(i);
        }
      }
      if (j < TS) break;  // no tile left, or a wait ran out
    }
    if (failed && lane == 0) atomicOr(a.status, STATUS_TIMEOUT);
    // before the CTA ends, the copies of the last stages issued must have landed
    for (int q = drain_first(s, NB); q < s; ++q)
        if (q != a.skip_stage) wait_phase(full0 + 8 * (q % NB), full_parity(q, NB), a.wait_limit);
    // the last CTA to draw its last ticket clears the counters for the next pass
    if (t == 0 && lane == 0) {
        __threadfence();
        if (atomicAdd(a.tickets + 1, 1u) == gridDim.x - 1) {
            a.tickets[0] = 0;
            a.tickets[1] = 0;
        }
    }
}

// ---------------------------------------------------------------- the consumers' column work
// A thread advances both types of one cell: lane x of a pair is the cos type, lane y the sin type.
// The packed operations issue one instruction for the two lanes.
RTPN_HD float2 pair_fma(float2 a, float2 b, float2 c) {
#ifdef __CUDA_ARCH__
    return __ffma2_rn(a, b, c);
#else
    return make_float2(fmaf(a.x, b.x, c.x), fmaf(a.y, b.y, c.y));
#endif
}
RTPN_HD float2 pair_mul(float2 a, float2 b) {
#ifdef __CUDA_ARCH__
    return __fmul2_rn(a, b);
#else
    return make_float2(a.x * b.x, a.y * b.y);
#endif
}
RTPN_HD float2 pair_sub(float2 a, float2 b) {
#ifdef __CUDA_ARCH__
    return __fadd2_rn(a, make_float2(-b.x, -b.y));
#else
    return make_float2(a.x - b.x, a.y - b.y);
#endif
}

// Byte offsets in a stage buffer of a cell's operands, fixed per tile: its source value (type 0; type
// 1 is SRC_T further), the y partner of each type, and per parity p of the source column the z
// partner (type 0; the types share its direction) and the x partner of each type (opposite
// directions).
struct Operands {
    int c, y[2], z[2], x[2][2];
};

// T: kept for host programs that walk a tile type by type; the offsets serve both types
template <int N, int A, typename S, int TX, int TY, int TZ, int NB, int NCH>
RTPN_HD Operands operand_offsets(const TileGeo& g, int /*T*/, int lx, int ly, int lz) {
    using L = Layout<N, A, S, TX, TY, TZ, NB, NCH>;
    constexpr int B = 1 - A, ES = L::ES, REG = L::REG;
    const int cp = (ly * TX + lx) * ES;  // the cell in a tile plane region (per component)
    Operands op;
    op.c = L::SRCO + lz * REG + cp;
#pragma unroll
    for (int t = 0; t < 2; ++t) {
        const int src = L::SRCO + t * L::SRC_T;
        const int dy = t == 0 ? 1 : -1;  // cos-type sources are read at y+1, sin-type at y-1
        op.y[t] = (ly + dy >= 0 && ly + dy < g.wy) ? op.c + t * L::SRC_T + dy * TX * ES
                                                   : src + L::KY * REG + (lz * TX + lx) * ES;
#pragma unroll
        for (int p = 0; p < 2; ++p) {
            const int dx = dir_x(p, t);
            op.x[p][t] = (lx + dx >= 0 && lx + dx < g.wx)
                             ? op.c + t * L::SRC_T + dx * ES
                             : src + L::KX * REG + ((lz * L::RY + ly) * L::XW + (dx > 0 ? g.hx_elem[1] : g.hx_elem[0])) * ES;
        }
    }
#pragma unroll
    for (int p = 0; p < 2; ++p) {
        const int dz = ((B + p) & 1) == 0 ? 1 : -1;
        op.z[p] = (lz + dz >= 0 && lz + dz < g.wz) ? op.c + dz * REG : L::SRCO + L::KZ * REG + cp;
    }
    return op;
}

// What a column's sweep reads beside the sources themselves: the x and y partners (cos, sin) and the z
// partner, as offsets in a stage buffer, and the factors of the y differences (the column's
// sign by target type, times sy).  At |m| = 0 the absent sin type's x and y differences are taken as
// zero: its partners are its own (stale) values.  src_t: offset between the types' regions.
struct ColumnOps {
    int x0, x1, y0, y1, z;
    float2 s;
};
RTPN_HD ColumnOps column_operands(const Operands& op, int i, int src_t, float sy) {
    const bool odd = i & 1;
    ColumnOps c;
    c.x0 = odd ? op.x[1][0] : op.x[0][0];
    c.x1 = odd ? op.x[1][1] : i == 0 ? op.c + src_t : op.x[0][1];
    c.y0 = op.y[0];
    c.y1 = i == 0 ? op.c + src_t : op.y[1];
    c.z = odd ? op.z[1] : op.z[0];
    c.s = odd ? make_float2(-sy, sy) : make_float2(sy, -sy);
    return c;
}

// One source slot's operands, both types: value, x, y and z partners, and its constants.
struct SlotOps {
    float c0, c1, x0, x1, y0, y1, z0, z1;
    float4 kz, ku, kd;  // pairs to l-1, l+1: of column M (z), M+1 and (negated) M-1 (x, and y unless SC)
    float4 kuy, kdy;    // SC: of y to M+1 and M-1
};

// Scatter the slots of sub-stage C of source column i (in a stage buffer) into the accumulators of target
// columns i - 1 (prev), i (cur) and i + 1 (next): every source value yields its half-grid differences
// (Section 2.1), each scattered into its <= 10 targets with the column's coupling constants (Eqs.
// 4-5).  At |m| = 0 only the cos type exists: the absent type's constants are zero or meet zero
// differences (its regions hold earlier, finite data), so the same sweep serves every column.  fq: the
// column's first source slot.
template <int N, int A, typename S, int TX, int TY, int TZ, int NB, int NCH, int C, bool SC = false>
RTPN_HD void sweep_pairs(const unsigned char* buf, int c0, const ColumnOps& op, int fq,
                         float2 (&prev)[(N - A) / 2 + 1], float2 (&cur)[(N - A) / 2 + 1],
                         float2 (&next)[(N - A) / 2 + 1]) {
    using L = Layout<N, A, S, TX, TY, TZ, NB, NCH>;
    constexpr int B = 1 - A, UB = L::UB, ST = L::SRC_T, K = L::K;
    constexpr int NLA = (N - A) / 2 + 1, NLB = (N - B) / 2 + 1;
    constexpr int KC = C * K + K <= NLB ? K : NLB - C * K;  // slots of this sub-stage
    const int skip = fq > C * K ? fq - C * K : 0;  // slots below the column's first source fq
    const unsigned char* bs = buf - skip * UB;     // slot k sits at k * UB from each base
    const unsigned char* pc = bs + c0;
    const unsigned char* pz = bs + op.z;
    const unsigned char* py0 = bs + op.y0;
    const unsigned char* py1 = bs + op.y1;
    const unsigned char* px0 = bs + op.x0;
    const unsigned char* px1 = bs + op.x1;
    const float4* kc = reinterpret_cast<const float4*>(buf + L::COEFO);
    auto load = [&](SlotOps& o, int k) {
        const int e = k * UB;
        o.c0 = lds<S>(pc, e);
        o.c1 = lds<S>(pc, e + ST);
        o.x0 = lds<S>(px0, e);
        o.x1 = lds<S>(px1, e);
        o.y0 = lds<S>(py0, e);
        o.y1 = lds<S>(py1, e);
        o.z0 = lds<S>(pz, e);
        o.z1 = lds<S>(pz, e + ST);
        constexpr int n4 = slot_pairs<SC>() / 2;
        RTPN_CHECK_PTR(kc + n4 * k + n4 - 1);
        o.kz = kc[n4 * k];
        o.ku = kc[n4 * k + 1];
        o.kd = kc[n4 * k + 2];
        if constexpr (SC) {
            o.kuy = kc[n4 * k + 3];
            o.kdy = kc[n4 * k + 4];
        }
    };
    auto work = [&](const SlotOps& o, auto ki) {
        constexpr int q = C * K + decltype(ki)::value;
        constexpr int ls = 2 * q + B;
        constexpr int lm = (ls - 1) / 2, lp = (ls + 1) / 2;  // acc index of l-1, l+1
        constexpr bool has_m = ls - 1 >= 0 && lm < NLA;
        constexpr bool has_p = ls + 1 <= N && lp < NLA;
        constexpr int am = has_m ? lm : 0, ap = has_p ? lp : 0;
        const float2 c = make_float2(o.c0, o.c1), xn = make_float2(o.x0, o.x1);
        const float2 dz = pair_sub(make_float2(o.z0, o.z1), c);
        const float2 dx = pair_sub(xn, c), nx = pair_sub(c, xn);
        const float2 dy = pair_mul(make_float2(o.y1 - o.c1, o.y0 - o.c0), op.s);  // the other type's
        if constexpr (has_m) cur[am] = pair_fma(make_float2(o.kz.x, o.kz.y), dz, cur[am]);
        if constexpr (has_p) cur[ap] = pair_fma(make_float2(o.kz.z, o.kz.w), dz, cur[ap]);
        if constexpr (has_m) prev[am] = pair_fma(make_float2(o.kd.x, o.kd.y), nx, prev[am]);
        if constexpr (has_p) prev[ap] = pair_fma(make_float2(o.kd.z, o.kd.w), nx, prev[ap]);
        if constexpr (has_m) next[am] = pair_fma(make_float2(o.ku.x, o.ku.y), dx, next[am]);
        if constexpr (has_p) next[ap] = pair_fma(make_float2(o.ku.z, o.ku.w), dx, next[ap]);
        const float4& kd = SC ? o.kdy : o.kd;
        const float4& ku = SC ? o.kuy : o.ku;
        if constexpr (has_m) prev[am] = pair_fma(make_float2(kd.x, kd.y), dy, prev[am]);
        if constexpr (has_p) prev[ap] = pair_fma(make_float2(kd.z, kd.w), dy, prev[ap]);
        if constexpr (has_m) next[am] = pair_fma(make_float2(ku.x, ku.y), dy, next[am]);
        if constexpr (has_p) next[ap] = pair_fma(make_float2(ku.z, ku.w), dy, next[ap]);
    };
    constexpr int NBLK = KC / kBlock > 0 ? KC / kBlock : 1;  // the last block takes the remainder
    static_for<NBLK>([&](auto bi) {
        constexpr int b0 = decltype(bi)::value * kBlock;
        constexpr int nb = decltype(bi)::value == NBLK - 1 ? KC - b0 : kBlock;
        if (b0 + nb > skip) {
            SlotOps o[nb];
            static_for<nb>([&](auto ki) { load(o[decltype(ki)::value], b0 + decltype(ki)::value); });
            static_for<nb>([&](auto ki) {
                work(o[decltype(ki)::value], std::integral_constant<int, b0 + decltype(ki)::value>{});
            });
        }
    });
}

#ifdef RTPN_HOST_CHECK
// The lane of type T of sweep_pairs over a whole column, for host programs that walk a tile type by type.
template <int N, int A, typename S, int TX, int TY, int TZ, int NB, int NCH>
RTPN_HD void sweep_column(const unsigned char* buf, const Operands& op, int T, int i,
                          float (&prev)[(N - A) / 2 + 1], float (&cur)[(N - A) / 2 + 1],
                          float (&next)[(N - A) / 2 + 1]) {
    using L = Layout<N, A, S, TX, TY, TZ, NB, NCH>;
    static_assert(NCH == 1, "one stage per column");
    constexpr int NLA = (N - A) / 2 + 1;
    float2 p[NLA], c[NLA], n[NLA];
    for (int q = 0; q < NLA; ++q) {
        p[q] = make_float2(prev[q], prev[q]);
        c[q] = make_float2(cur[q], cur[q]);
        n[q] = make_float2(next[q], next[q]);
    }
    sweep_pairs<N, A, S, TX, TY, TZ, NB, NCH, 0>(buf, op.c, column_operands(op, i, L::SRC_T, 1.f),
                                                first_source<N, A>(i), p, c, n);
    for (int q = 0; q < NLA; ++q) {
        prev[q] = T ? p[q].y : p[q].x;
        cur[q] = T ? c[q].y : c[q].x;
        next[q] = T ? n[q].y : n[q].x;
    }
}
#endif

// Finish the slots of target column M that sub-stage C completes, both types (accumulators in prev),
// from their old values in the stage's target planes (at byte offset tgo for this cell; the sin type
// TGT_T further) into global memory: FORWARD by Eq. (5), u' = alpha u + scale acc with scale = -beta / h
// (the u_0 factors al0, be0, ga0 for slot 0 of column 0, cos type, class 0); ADJ_SOURCES lam' = alpha
// lam + scale acc with scale = 1 / h (alpha = 1 when no factors are given).  q0: the column's first
// slot; t0, t1: slot q = 0 of the cos and the sin run at this cell, slots vb bytes apart; cos_t,
// sin_t: whether this cell's values of the type are stored.
template <int N, int A, typename S, int TX, int TY, int TZ, int NB, int NCH, int MODE, int C>
RTPN_HD void finish_pairs(const unsigned char* buf, int tgo, int M, int q0, char* t0, char* t1, unsigned vb, bool cos_t,
                          bool sin_t, float2 alpha, float2 scale, float al0, float be0, float ga0,
                          const float2 (&prev)[(N - A) / 2 + 1]) {
    using L = Layout<N, A, S, TX, TY, TZ, NB, NCH>;
    constexpr int UB = L::UB;
    constexpr int LO = window_lo<N, A, NCH>(C), HI = window_hi<N, A, NCH>(C);
    const int qs = q0 > LO ? q0 : LO;  // the slot the target boxes start with
    const unsigned char* ob = buf + tgo - (qs - LO) * UB;
    constexpr int kGroup = 3;
    constexpr int NG = (HI - LO + kGroup - 1) / kGroup;
    static_for<NG>([&](auto gi) {
        constexpr int g0 = LO + decltype(gi)::value * kGroup;
        constexpr int ng = g0 + kGroup <= HI ? kGroup : HI - g0;
        if (g0 + ng > qs) {
            float2 old[ng];
            static_for<ng>([&](auto ki) {
                constexpr int k = decltype(ki)::value, q = g0 + k;
                old[k] = make_float2(0.f, 0.f);
                if (k == ng - 1 || q >= qs)
                    old[k] = make_float2(lds<S>(ob, (q - LO) * UB), lds<S>(ob, (q - LO) * UB + L::TGT_T));
            });
            static_for<ng>([&](auto ki) {
                constexpr int k = decltype(ki)::value, q = g0 + k;
                // the product with the accumulator is rounded first in a forward pass, the one with the old
                // value in the adjoint's
                float2 nv = MODE == ADJ_SOURCES ? pair_fma(scale, prev[q], pair_mul(alpha, old[k]))
                                                : pair_fma(alpha, old[k], pair_mul(scale, prev[q]));
                if constexpr (A == 0 && q == 0)  // u_0
                    if (M == 0)
                        nv.x = MODE == ADJ_SOURCES ? fmaf(scale.x, prev[q].x, al0 * old[k].x)
                                                   : fmaf(al0, old[k].x, fmaf(-be0, prev[q].x, ga0));
                const bool in = k == ng - 1 || q >= qs;
                if (in && cos_t) win::store<S>(reinterpret_cast<S*>(t0 + (unsigned long long)q * vb), nv.x);
                if (in && sin_t) win::store<S>(reinterpret_cast<S*>(t1 + (unsigned long long)q * vb), nv.y);
            });
        }
    });
}

#ifdef RTPN_HOST_CHECK
// The same for type T alone over a whole column (accumulators, factors and the run's first component
// tp of that type), for host programs that walk a tile type by type.
template <int N, int A, typename S, int TX, int TY, int TZ, int NB, int NCH, int MODE>
RTPN_HD void finish_column(const unsigned char* buf, int tgo, int M, int T, S* tp, long long V, bool active,
                           float alpha, float beta, float al0, float be0, float ga0, float inv_h,
                           const float (&prev)[(N - A) / 2 + 1]) {
    using L = Layout<N, A, S, TX, TY, TZ, NB, NCH>;
    static_assert(NCH == 1, "one stage per column");
    constexpr int NLA = (N - A) / 2 + 1;
    float2 p[NLA];
    for (int q = 0; q < NLA; ++q) p[q] = make_float2(prev[q], prev[q]);
    const float scale = MODE == ADJ_SOURCES ? inv_h : -beta;
    finish_pairs<N, A, S, TX, TY, TZ, NB, NCH, MODE, 0>(
        buf, tgo - T * L::TGT_T, M, first_l(M, A) / 2, reinterpret_cast<char*>(tp), reinterpret_cast<char*>(tp),
        (unsigned)(V * (long long)sizeof(S)), active && T == 0, active && T == 1, make_float2(alpha, alpha),
        make_float2(scale, scale), al0, be0, ga0, p);
}
#endif

template <int N, int A, typename S, int TX, int TY, int TZ, int NB, int NCH, int MODE, bool SC>
__device__ __forceinline__ void stage_kernel_body(const Args& a, unsigned char* smem) {
    using L = Layout<N, A, S, TX, TY, TZ, NB, NCH, SC>;
    static_assert(N >= 1, "order N >= 1");
    static_assert(L::NMAP <= kMaxSlots, "tensor maps of a kind");
    constexpr int B = 1 - A;
    constexpr int NLA = (N - A) / 2 + 1;   // class-A components of a run, at most
    constexpr int ES = L::ES;
    constexpr int NST = N + 2;  // stage i: sources of column i (i <= N), targets of column i - 1
    const int cA0 = A == 0 ? 0 : class_size(N, 0);
    [[maybe_unused]] const int* colA = a.colstart + A * (N + 2);
    const int tid = threadIdx.x;
    const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;  // warp: uniform for the compiler
    const long long V = a.V;

    // TMA writes into shared memory need 128-byte aligned destinations; the dynamic shared memory
    // window is not guaranteed to start on one, so the layout starts at the next 128-byte boundary.
    smem += (128u - (smem_addr(smem) & 127u)) & 127u;
    // zero the ring once: slots a chunked sweep reads below a column's first source
    // (with zero coupling constants) then always hold finite values
    for (int k = tid; k < NB * L::BUF / 16; k += blockDim.x)
        reinterpret_cast<uint4*>(smem)[k] = make_uint4(0u, 0u, 0u, 0u);
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // before the TMA writes the ring
    unsigned char* bufs = smem;
    unsigned long long* bars = reinterpret_cast<unsigned long long*>(bufs + NB * L::BUF);
    const unsigned full0 = smem_addr(&bars[0]), empty0 = smem_addr(&bars[NB]);
    volatile unsigned* next = reinterpret_cast<unsigned*>(bufs + NB * L::BUF + L::BARS);
    if (tid < kNextRing) next[tid] = 0xffffffffu;  // no tile
    if (tid == 0) {
        for (int b = 0; b < NB; ++b) {
            mbar_init(full0 + 8 * b, kProducers);  // each producer's arrive.expect_tx
            mbar_init(empty0 + 8 * b, L::CONSUMER_WARPS);
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();

    if (warp >= L::CONSUMER_WARPS) {
        stage_producer<N, A, S, TX, TY, TZ, NB, NCH, SC>(a, bufs, full0, empty0, next, warp - L::CONSUMER_WARPS);
        return;
    }

    // ---- consumers: a thread finishes the targets of both types in its cell
    const int lx = tid % TX, ly = (tid / TX) % TY, lz = tid / (TX * TY);
    const int tgo = L::TGTO + lz * L::REGT + (ly * TX + lx) * ES;  // this cell's old target values (type 0)

    // the three live target columns; their roles (prev, cur, next) rotate by one per stage
    float2 wa[NLA], wb[NLA], wc[NLA];

    const unsigned vb = (unsigned)(a.sV * ES);  // bytes of a component of the target array
    unsigned limit = a.wait_limit;           // 0 once a wait has run out: the rest of the pass is not waited for
    unsigned tile = blockIdx.x;
    unsigned b = 0, ph = 0;                  // stage buffer, phase parity of its current use
    // tile after tile until none is left (a consumer whose wait ran out leaves after the tile it is on)
    for (unsigned k = 0; k == 0 || limit != 0; ++k) {
        if (k > 0) tile = next[k % kNextRing];
        if (tile >= (unsigned long long)a.tiles) break;
        const TileGeo g = tile_geo<TX, TY, TZ, L::G>(a, tile);
        const bool active = lx < g.wx && ly < g.wy && lz < g.wz;
        const long long cell = ((long long)(g.z0 + lz) * a.ny + (g.y0 + ly)) * a.nx + (g.x0 + lx);
        const Operands op = operand_offsets<N, A, S, TX, TY, TZ, NB, NCH>(g, 0, lx, ly, lz);  // fixed per tile
        float2 al[2] = {}, be[2] = {};         // Eq. (5) factors by parity of M
        float al0 = 0.f, be0 = 0.f, ga0 = 0.f; // u_0 (class 0, type 0 only)
        if (active && (MODE == FORWARD || a.fac)) {  // ADJ_SOURCES: the alphas only, if asked
            // sub-grid slot of (l, M, T) in class A: x by (M, T), y by T, z by (A + M)
#pragma unroll
            for (int par = 0; par < 2; ++par) {
                const int gz = ((A + par) & 1) == 0 ? 0 : 1;
                const int gc = (par == 0 ? 0 : 1) + 4 * gz, gs = (par == 0 ? 1 : 0) + 2 + 4 * gz;
                const float* f = a.fac + (long long)a.fac_ofs * V + cell;
                al[par] = make_float2(__ldg(f + 2 * gc * V), __ldg(f + 2 * gs * V));
                if (MODE == FORWARD) be[par] = make_float2(__ldg(f + (2 * gc + 1) * V), __ldg(f + (2 * gs + 1) * V));
            }
            if (A == 0) {
                al0 = __ldg(a.fac + (long long)FAC_U0 * V + cell);
                be0 = __ldg(a.fac + (long long)(FAC_U0 + 1) * V + cell);
                ga0 = __ldg(a.fac + (long long)(FAC_U0 + 2) * V + cell);
            }
        } else if (MODE == ADJ_SOURCES) {
            al[0] = al[1] = make_float2(1.f, 1.f);
            al0 = 1.f;
        }
#pragma unroll
        for (int q = 0; q < NLA; ++q) wa[q] = wb[q] = wc[q] = make_float2(0.f, 0.f);
        char* const tcell = reinterpret_cast<char*>(a.tgt) +
                            (((long long)(g.z0 + lz) * a.ny + (g.y0 + ly)) * a.px + (g.x0 + lx)) * ES;
        unsigned comp = cA0;  // the first component of target column M in the target array

        // One column: its sub-stages sweep source column i into prev (column i - 1), cur (i) and next
        // (i + 1) and finish prev slot by slot; then prev is cleared (it is the next column's `next`).
        auto column = [&](int i, float2 (&prev)[NLA], float2 (&cur)[NLA], float2 (&next)[NLA]) {
            const int C0 = first_chunk<N, A, NCH>(i), fq = first_source<N, A>(i);
            const bool sources = i <= N && 2 * fq + B <= N;
            const ColumnOps cop = column_operands(op, i, L::SRC_T, a.sy);
            // target column M = i - 1
            const int M = i - 1, q0 = M >= 0 ? first_source<N, B>(M) : 0, lenA = NLA - q0;
            (void)RTPN_SCHECK(M < 0 || comp == (unsigned)(cA0 + colA[M]));
            char* const t0 = tcell + (unsigned long long)(comp - (unsigned)q0) * vb;
            char* const t1 = t0 + (unsigned long long)(unsigned)lenA * vb;
            const bool odd = M & 1, sin_t = active && M >= 1;
            const float2 alpha = odd ? al[1] : al[0];
            const float2 scale = MODE == ADJ_SOURCES ? make_float2(a.inv_h, a.inv_h)
                                                     : pair_mul(odd ? be[1] : be[0], make_float2(-a.inv_h, -a.inv_h));
            static_for<NCH>([&](auto ci) {
                constexpr int C = decltype(ci)::value;
                if (C < C0) return;
                if (!wait_phase(full0 + 8 * b, ph, limit)) {
                    if (lane == 0) atomicOr(a.status, STATUS_TIMEOUT);
                    limit = 0;
                }
                const unsigned char* buf = bufs + b * (unsigned)L::BUF;
                // the sweep and the finish run on every thread of the tile (a thread past the grid's edge
                // works on zero-filled or in-tile shared memory), only global accesses need an active cell
                if (sources) sweep_pairs<N, A, S, TX, TY, TZ, NB, NCH, C, SC>(buf, op.c, cop, fq, prev, cur, next);
                if (M >= 0)
                    finish_pairs<N, A, S, TX, TY, TZ, NB, NCH, MODE, C>(buf, tgo, M, q0, t0, t1, vb, active, sin_t, alpha,
                                                                        scale, al0, be0 * a.inv_h, ga0, prev);
                // the stage buffer is free once every lane of the warp is past its reads
                __syncwarp();
                if (lane == 0 && hands_back(limit)) mbar_arrive(empty0 + 8 * b);
                if (++b == NB) {
                    b = 0;
                    ph ^= 1u;
                }
            });
#pragma unroll
            for (int q = 0; q < NLA; ++q) prev[q] = make_float2(0.f, 0.f);
            if (M >= 0) comp += (unsigned)((M >= 1 ? 2 : 1) * lenA);
        };
        // unrolled by three: the window's roles rotate instead of its registers moving
        for (int i = 0; i < NST; i += 3) {
            column(i, wa, wb, wc);
            if (NST % 3 == 0 || i + 1 < NST) column(i + 1, wb, wc, wa);
            if (NST % 3 == 0 || i + 2 < NST) column(i + 2, wc, wa, wb);
        }
    }
}

}  // namespace stg
}  // namespace rtpn
