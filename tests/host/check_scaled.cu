// Host check of the staged kernel's form SC (test program): the sweep of every sub-stage of every column over a
// random stage buffer, against a scalar loop with one FP32 constant per (source, relation), the y ones
// rounded once from the coupling times h / h_y: bit for bit.  With h / h_y = 1 the form's sums are also those
// of the plain form.
//
// Compile with -DRTPN_SN=<order> -DRTPN_STX= -DRTPN_STY= -DRTPN_STZ= -DRTPN_SNB= -DRTPN_SEM=<sub-stages>.
// usage: check_scaled h/h_y h/h_z seed; prints the values compared, those that differ, and those of the plain form
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <random>
#include <vector>

#include "stage_impl.cuh"

using namespace rtpn;
using namespace rtpn::stg;

constexpr int kN = RTPN_SN, kTX = RTPN_STX, kTY = RTPN_STY, kTZ = RTPN_STZ, kNB = RTPN_SNB, kCH = RTPN_SEM;

static long long g_seen = 0, g_bad = 0, g_bad_plain = 0;

static bool same(float a, float b) { return std::memcmp(&a, &b, 4) == 0 || (a == 0.f && b == 0.f); }

template <int A>
void check(const Model& md, double sy, double sz, unsigned seed) {
    using L = Layout<kN, A, float, kTX, kTY, kTZ, kNB, kCH, true>;
    using LP = Layout<kN, A, float, kTX, kTY, kTZ, kNB, kCH>;
    static_assert(L::COEFO == LP::COEFO && L::SRCO == LP::SRCO, "the forms share the regions");
    constexpr int B = 1 - A, NLA = (kN - A) / 2 + 1, NLB = (kN - B) / 2 + 1, UB = L::UB;
    std::vector<int> col;
    std::vector<float> tab[2], plain[2], t10;
    if (!coupling_tables(md, sy, sz, tab, &col, true) || !coupling_tables(md, 1.0, sz, plain, &col) ||
        !win::coef_table(md, A, &t10))
        std::exit(3);
    std::mt19937 rng(seed);
    std::normal_distribution<float> dist;
    std::vector<float> store(L::BUF / 4 + 64);
    unsigned char* buf = reinterpret_cast<unsigned char*>(store.data());
    TileGeo g{};
    g.wx = kTX;
    g.wy = kTY;
    g.wz = kTZ;
    const Operands op = operand_offsets<kN, A, float, kTX, kTY, kTZ, kNB, kCH>(g, 0, 7, 0, 1);
    for (int i = 0; i <= kN; ++i)
        static_for<kCH>([&](auto ci) {
            constexpr int C = decltype(ci)::value;
            if (C < first_chunk<kN, A, kCH>(i)) return;
            const int fq = first_source<kN, A>(i);
            if (2 * fq + B > kN) return;
            for (int k = 0; k < L::COEFO / 4; ++k) store[k] = dist(rng);
            auto constants = [&](const std::vector<float>& t, int pairs) {
                const float* src = t.data() + (size_t)(i * L::NLC + C * L::K) * 2 * pairs;
                std::memcpy(buf + L::COEFO, src, (size_t)coef_slots<kN, kCH>(C) * 2 * pairs * 4);
            };
            float2 w[3][NLA], p[3][NLA], r[3][NLA];
            for (auto& x : w)
                for (auto& v : x) v = make_float2(dist(rng), dist(rng));
            std::memcpy(p, w, sizeof w);
            std::memcpy(r, w, sizeof w);
            const ColumnOps cop = column_operands(op, i, L::SRC_T, 1.f);
            constants(plain[A], KPAIRS);
            sweep_pairs<kN, A, float, kTX, kTY, kTZ, kNB, kCH, C>(buf, op.c, cop, fq, p[0], p[1], p[2]);
            constants(tab[A], L::PAIRS);
            sweep_pairs<kN, A, float, kTX, kTY, kTZ, kNB, kCH, C, true>(buf, op.c, cop, fq, w[0], w[1], w[2]);
            const int first = fq > C * L::K ? fq : C * L::K, skip = fq > C * L::K ? fq - C * L::K : 0;
            for (int q = first; q < C * L::K + L::K && q < NLB; ++q) {
                const int at = (q - C * L::K - skip) * UB, l = 2 * q + B, len = column_len(kN, i, B);
                auto val = [&](int ofs) { return *reinterpret_cast<const float*>(buf + ofs + at); };
                for (int T = 0; T < 2; ++T) {
                    auto rel = [&](int t) -> const float* {
                        return t < ntypes(i) ? &t10[(size_t)(col[B * (kN + 2) + i] + t * len + q - fq) * 10] : nullptr;
                    };
                    const float *own = rel(T), *oth = rel(1 - T);
                    const float dz = val(op.z[i & 1] + T * L::SRC_T) - val(op.c + T * L::SRC_T);
                    const float dx = val(op.x[i & 1][T]) - val(op.c + T * L::SRC_T);
                    const float dy = val(op.y[1 - T]) - val(op.c + (1 - T) * L::SRC_T);
                    auto acc = [&](int c, int j) -> float* {
                        if (j < 0 || j >= NLA) return nullptr;
                        return T ? &r[c][j].y : &r[c][j].x;
                    };
                    auto add = [&](int c, const float* k, double scale, float d) {
                        for (int s = 0; s < 2 && k; ++s) {
                            const int lt = l + (s ? 1 : -1);
                            float* a = lt < 0 || lt > kN ? nullptr : acc(c, (lt - A) / 2);
                            if (a) *a = std::fmaf((float)(k[s] * scale), d, *a);
                        }
                    };
                    add(1, own, sz, dz);
                    add(0, own ? own + 2 : nullptr, 1.0, dx);
                    add(2, own ? own + 4 : nullptr, 1.0, dx);
                    add(0, oth ? oth + 6 : nullptr, sy, dy);
                    add(2, oth ? oth + 8 : nullptr, sy, dy);
                }
            }
            for (int c = 0; c < 3; ++c)
                for (int j = 0; j < NLA; ++j) {
                    g_seen += 2;
                    g_bad += !same(w[c][j].x, r[c][j].x) + !same(w[c][j].y, r[c][j].y);
                    g_bad_plain += !same(w[c][j].x, p[c][j].x) + !same(w[c][j].y, p[c][j].y);
                }
        });
}

int main(int argc, char** argv) {
    if (argc < 4) return 2;
    const Model md = build_model(kN);
    check<0>(md, atof(argv[1]), atof(argv[2]), (unsigned)atoi(argv[3]));
    check<1>(md, atof(argv[1]), atof(argv[2]), (unsigned)atoi(argv[3]) + 1);
    printf("%lld %lld %lld\n", g_seen, g_bad, g_bad_plain);
    return 0;
}
