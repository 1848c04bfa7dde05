// Host run of the TMA-staged substep kernel with several sub-stages per column (test program): the
// kernel's own sub-stage plan (stg::stage_runs, stg::stage_box, stg::stage_bytes) and column work
// (stg::operand_offsets, stg::sweep_pairs, stg::finish_pairs) compiled for the host, CTA by CTA in the
// kernel's tile walk over bounds-checked memory, both types of a cell together as on the device.  The
// boxes are copied as the TMA unit copies them; the program aborts on a box that leaves its region, an
// unaligned x coordinate or destination, a byte count that differs from the expected one, and on any
// access outside the ring, the state, the coupling constants or the factor planes.
//
// Compile with -DRTPN_SN=<order> -DRTPN_STX= -DRTPN_STY= -DRTPN_STZ= -DRTPN_SNB= -DRTPN_SEM=<sub-stages>.
// usage: as emulate_stage (without the adjoint's modes), and a last argument h/h_y of the y differences
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <string>
#include <vector>

static const char* g_lo[8];
static const char* g_hi[8];
static int g_nr = 0;
static void check_ptr(const void* p) {
    const char* c = (const char*)p;
    for (int i = 0; i < g_nr; ++i)
        if (c >= g_lo[i] && c < g_hi[i]) return;
    fprintf(stderr, "OUT OF BOUNDS access %p\n", p);
    std::abort();
}
static void fail(const char* what, long long v) {
    fprintf(stderr, "STAGE PLAN ERROR: %s (%lld)\n", what, v);
    std::abort();
}
#define RTPN_HOST_CHECK 1
#define RTPN_CHECK_PTR(p) check_ptr(p)
#include "stage_impl.cuh"

using namespace rtpn;
using namespace rtpn::stg;

constexpr int kN = RTPN_SN, kTX = RTPN_STX, kTY = RTPN_STY, kTZ = RTPN_STZ, kNB = RTPN_SNB, kCH = RTPN_SEM;

template <int A, typename S>
void run(const Args& a, const float* fac, S* u, const std::vector<float>& coef, int sms) {
    using L = Layout<kN, A, S, kTX, kTY, kTZ, kNB, kCH>;
    constexpr int B = 1 - A, NST = kN + 2, NLA = (kN - A) / 2 + 1, CELLS = L::CELLS;
    constexpr int NJOB = 2 * L::NKIND + 2 * kTZ;
    if (!L::FITS) fail("variant does not fit this storage", 0);
    const long long V = a.V;
    const int cA0 = A == 0 ? 0 : class_size(kN, 0), nc = class_size(kN, 0) + class_size(kN, 1);
    const long long grid = a.tiles < sms ? a.tiles : sms;
    std::vector<unsigned char> ring((size_t)kNB * L::BUF);
    g_lo[3] = (const char*)ring.data();
    g_hi[3] = (const char*)(ring.data() + ring.size());
    std::vector<float2> win((size_t)CELLS * 3 * NLA);
    for (long long cta = 0; cta < grid; ++cta) {
        std::fill(ring.begin(), ring.end(), 0);
        long long s = 0;
        for (long long tile = cta; tile < a.tiles; tile += grid) {
            const TileGeo g = tile_geo<kTX, kTY, kTZ, L::G>(a, (unsigned)tile);
            std::fill(win.begin(), win.end(), make_float2(0.f, 0.f));
            int offA = 0, offB = 0, rot = 0, stages = 0;
            for (int i = 0; i < NST; ++i) {
                const int fq = first_source<kN, A>(i), M = i - 1, q0 = M >= 0 ? first_l(M, A) / 2 : 0;
                if (fq != first_l(i, B) / 2) fail("first source", i);
                for (int C = first_chunk<kN, A, kCH>(i); C < kCH; ++C, ++s, ++stages) {
                    unsigned char* buf = ring.data() + (size_t)(s % kNB) * L::BUF;
                    const StageRuns r = stage_runs<kN, A, kCH>(i, C);
                    unsigned landed = 0;
                    for (int j = 0; j < NJOB; ++j) {
                        const BoxJob bj = stage_box<kN, A, S, kTX, kTY, kTZ, kNB, kCH>(a, g, i, r, offA, offB, j);
                        if (!bj.valid) continue;
                        const int E = bj.emap + 1;
                        int bx = kTX, by = kTY, bz = 1;
                        if (!bj.target && bj.kind == MAP_YROW) by = 1, bz = kTZ;
                        if (!bj.target && bj.kind == MAP_XGRP) bx = L::XW, by = L::RY, bz = kTZ;
                        const int base = bj.target ? L::TGTO : L::SRCO, reg = bj.target ? L::REGT : L::REG;
                        const int end = (bj.dst - base) / reg * reg + reg + base;
                        const long long bytes = (long long)E * bx * by * bz * L::ES;
                        if (bytes != (long long)E * L::UB) fail("box volume", bytes);
                        if (bj.dst % 128 != 0) fail("destination", bj.dst);
                        if (bj.dst + bytes > end || end > L::COEFO) fail("box leaves its region", bj.dst);
                        if (((long long)bj.x * L::ES) % 16 != 0) fail("x coordinate", bj.x);
                        if (E < 1 || E > L::NMAP) fail("box length", E);
                        for (int ec = 0; ec < E; ++ec)
                            for (int ez = 0; ez < bz; ++ez)
                                for (int ey = 0; ey < by; ++ey)
                                    for (int ex = 0; ex < bx; ++ex) {
                                        const long long X = bj.x + ex, Y = bj.y + ey, Z = bj.z + ez, c = bj.c + ec;
                                        S v{};
                                        if (X >= 0 && X < a.nx && Y >= 0 && Y < a.ny && Z >= 0 && Z < a.nz && c >= 0 && c < nc) {
                                            check_ptr(u + c * V + (Z * a.ny + Y) * a.nx + X);
                                            v = u[c * V + (Z * a.ny + Y) * a.nx + X];
                                        }
                                        S* d = reinterpret_cast<S*>(buf + bj.dst) + (((ec * bz + ez) * by + ey) * bx + ex);
                                        check_ptr(d);
                                        *d = v;
                                    }
                        landed += (unsigned)bytes;
                    }
                    if (r.nt > 0) {
                        const int n = coef_slots<kN, kCH>(C) * 2 * CPAD;
                        const float* src = coef.data() + (size_t)(i * L::NLC + C * L::K) * (2 * CPAD);
                        check_ptr(src);
                        check_ptr(src + n - 1);
                        std::copy(src, src + n, reinterpret_cast<float*>(buf + L::COEFO));
                        landed += n * 4;
                    }
                    if (landed != stage_bytes<kN, A, S, kTX, kTY, kTZ, kNB, kCH>(r, C)) fail("expected bytes", landed);
                    for (int tid = 0; tid < CELLS; ++tid) {
                        const int lx = tid % kTX, ly = (tid / kTX) % kTY, lz = tid / (kTX * kTY);
                        float2* W = &win[(size_t)tid * 3 * NLA];
                        float2(&prev)[NLA] = *reinterpret_cast<float2(*)[NLA]>(W + rot * NLA);
                        float2(&cur)[NLA] = *reinterpret_cast<float2(*)[NLA]>(W + (rot + 1) % 3 * NLA);
                        float2(&next)[NLA] = *reinterpret_cast<float2(*)[NLA]>(W + (rot + 2) % 3 * NLA);
                        const Operands op = operand_offsets<kN, A, S, kTX, kTY, kTZ, kNB, kCH>(g, 0, lx, ly, lz);
                        const ColumnOps cop = column_operands(op, i, L::SRC_T, a.sy);
                        const bool active = lx < g.wx && ly < g.wy && lz < g.wz;
                        const long long cell = ((long long)(g.z0 + lz) * a.ny + (g.y0 + ly)) * a.nx + (g.x0 + lx);
                        float f[2][2] = {}, f0[3] = {};
                        if (active && M >= 0) {
                            for (int T = 0; T < 2; ++T) {
                                const int gx = ((M & 1) == 0) == (T == 0) ? 0 : 1, gz = ((A + M) & 1) == 0 ? 0 : 1;
                                for (int k = 0; k < 2; ++k) f[k][T] = fac[(long long)(a.fac_ofs + 2 * (gx + 2 * T + 4 * gz) + k) * V + cell];
                            }
                            for (int k = 0; k < 3; ++k) f0[k] = fac[(long long)(FAC_U0 + k) * V + cell];
                        }
                        const int tgo = L::TGTO + lz * L::REGT + (ly * kTX + lx) * L::ES;
                        char* t0 = reinterpret_cast<char*>(u + (cA0 + offA - q0) * V + cell);
                        char* t1 = t0 + (long long)(M >= 0 ? column_len(kN, M, A) : 0) * V * L::ES;
                        static_for<kCH>([&](auto ci) {
                            constexpr int CC = decltype(ci)::value;
                            if (CC != C) return;
                            if (column_len(kN, i, B) > 0)
                                sweep_pairs<kN, A, S, kTX, kTY, kTZ, kNB, kCH, CC>(buf, op.c, cop, fq, prev, cur, next);
                            if (M >= 0)
                                finish_pairs<kN, A, S, kTX, kTY, kTZ, kNB, kCH, FORWARD, CC>(
                                    buf, tgo, M, q0, t0, t1, (unsigned)(V * L::ES), active, active && M >= 1,
                                    make_float2(f[0][0], f[0][1]), make_float2(-f[1][0] * a.inv_h, -f[1][1] * a.inv_h), f0[0],
                                    f0[1] * a.inv_h, f0[2], prev);
                        });
                        if (C == kCH - 1) std::fill(prev, prev + NLA, make_float2(0.f, 0.f));
                    }
                }
                rot = (rot + 1) % 3;
                offB += ntypes(i) * column_len(kN, i, B);
                if (i >= 1) offA += ntypes(i - 1) * column_len(kN, i - 1, A);
            }
            if (stages != tile_stages<kN, A, kCH>()) fail("stages of a tile", stages);
        }
    }
}

int main(int argc, char** argv) {
    if (argc < 13) {
        fprintf(stderr, "usage\n");
        return 2;
    }
    const int A = atoi(argv[1]), nx = atoi(argv[2]), ny = atoi(argv[3]), nz = atoi(argv[4]), bc = atoi(argv[5]);
    const double h = atof(argv[6]), dt = atof(argv[7]);
    const int half = atoi(argv[8]);
    const std::string prec = argv[9];
    const int sms = atoi(argv[10]);
    const char* inf = argv[11];
    const char* outf = argv[12];
    const double sy = argc > 13 ? atof(argv[13]) : 1.0;
    const int N = kN;
    Model md = build_model(N);
    const long long V = (long long)nx * ny * nz;
    const int narr = 1;
    std::vector<double> in((size_t)(narr * md.nc + 3) * V);
    FILE* f = fopen(inf, "rb");
    if (!f || fread(in.data(), 8, in.size(), f) != in.size()) {
        fprintf(stderr, "bad input\n");
        return 4;
    }
    fclose(f);
    const double* sa = in.data() + (size_t)narr * md.nc * V;
    const double* ss = sa + V;
    const double* q = ss + V;
    // factor planes by the rule of rtpn_set_media (mean of sigma over the cells adjacent to a
    // sub-grid point; alpha = exp(-c tau), beta = tau E(-c tau)), FP32
    std::vector<float> fac((size_t)FAC_PLANES * V);
    auto idx = [&](int x, int y, int z) { return ((long long)z * ny + y) * nx + x; };
    for (int z = 0; z < nz; ++z)
        for (int y = 0; y < ny; ++y)
            for (int x = 0; x < nx; ++x) {
                const long long cell = idx(x, y, z);
                for (int code = 0; code < 8; ++code) {
                    const int gx = code & 1, gy = (code >> 1) & 1, gz = (code >> 2) & 1;
                    double sum = 0;
                    int cnt = 0;
                    for (int dz = 0; dz <= gz; ++dz)
                        for (int dy = 0; dy <= gy; ++dy)
                            for (int dx = 0; dx <= gx; ++dx) {
                                int xx = x + dx, yy = y + dy, zz = z + dz;
                                if (xx >= nx || yy >= ny || zz >= nz) {
                                    if (bc) continue;
                                    xx %= nx;
                                    yy %= ny;
                                    zz %= nz;
                                }
                                const long long j = idx(xx, yy, zz);
                                sum += sa[j] + ss[j];
                                ++cnt;
                            }
                    const double c = sum / cnt;
                    for (int hh = 0; hh < 2; ++hh) {
                        const double tau = hh ? 0.5 * dt : dt;
                        const double al = exp(-c * tau), be = c != 0 ? -expm1(-c * tau) / c : tau;
                        fac[(size_t)((hh ? FAC_HALF : FAC_FULL) + 2 * code) * V + cell] = (float)al;
                        fac[(size_t)((hh ? FAC_HALF : FAC_FULL) + 2 * code + 1) * V + cell] = (float)be;
                    }
                }
                const double c = sa[cell], al = exp(-c * dt), be = c != 0 ? -expm1(-c * dt) / c : dt;
                fac[(size_t)FAC_U0 * V + cell] = (float)al;
                fac[(size_t)(FAC_U0 + 1) * V + cell] = (float)be;
                fac[(size_t)(FAC_U0 + 2) * V + cell] = (float)(be * q[cell]);
            }
    std::vector<int> col;
    std::vector<float> tab[2];
    if (!coupling_tables(md, sy, 1.0, tab, &col)) {
        fprintf(stderr, "coupling tables\n");
        return 3;
    }
    Args a{};
    a.V = V;
    a.nx = nx;
    a.ny = ny;
    a.nz = nz;
    a.bc = bc;
    a.fac_ofs = half ? FAC_HALF : FAC_FULL;
    a.inv_h = (float)(1.0 / h);
    a.sy = (float)sy;
    a.ntx = (nx + kTX - 1) / kTX;
    a.nty = (ny + kTY - 1) / kTY;
    a.ntz = (nz + kTZ - 1) / kTZ;
    a.tiles = (long long)a.ntx * a.nty * a.ntz;
    {
        const double side = std::sqrt((double)sms / a.ntx);
        const int kz = (int)(side + 0.5);
        a.kz = kz < 1 ? 1 : (kz > a.ntz ? a.ntz : kz);
    }
    a.src_c0 = A == 1 ? 0 : md.ne;  // the source class is the other one
    a.nc = md.nc;
    g_lo[0] = (const char*)fac.data();
    g_hi[0] = (const char*)(fac.data() + fac.size());
    g_lo[1] = (const char*)tab[A].data();
    g_hi[1] = (const char*)(tab[A].data() + tab[A].size());
    std::vector<double> out((size_t)md.nc * V);
    auto go = [&](auto tag) {
        using S = decltype(tag);
        std::vector<S> u((size_t)md.nc * V);
        for (int c = 0; c < md.nc; ++c)
            for (long long i = 0; i < V; ++i) {
                const double v = in[(size_t)c * V + i];
                if constexpr (sizeof(S) == 4)
                    u[(size_t)md.internal_of_abi[c] * V + i] = (float)v;
                else
                    u[(size_t)md.internal_of_abi[c] * V + i] = __float2bfloat16_rn((float)v);
            }
        g_lo[2] = (const char*)u.data();
        g_hi[2] = (const char*)(u.data() + u.size());
        g_nr = 4;
        if (A == 0)
            run<0, S>(a, fac.data(), u.data(), tab[0], sms);
        else
            run<1, S>(a, fac.data(), u.data(), tab[1], sms);
        for (int c = 0; c < md.nc; ++c)
            for (long long i = 0; i < V; ++i) {
                const S v = u[(size_t)md.internal_of_abi[c] * V + i];
                if constexpr (sizeof(S) == 4)
                    out[(size_t)c * V + i] = v;
                else
                    out[(size_t)c * V + i] = __bfloat162float(v);
            }
    };
    if (prec == "fp32")
        go(float{});
    else
        go(__nv_bfloat16{});
    f = fopen(outf, "wb");
    fwrite(out.data(), 8, out.size(), f);
    fclose(f);
    return 0;
}
