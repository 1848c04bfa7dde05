// Host model of the staged kernel's ring of stage buffers (test program): the full and empty barriers of one
// CTA, its two producers and its consumer warps, advanced one at a time in a random order, with copies
// that land at random times and waits that give up after a number of polls.  The agents follow
// stage_producer and the consumers' loop of stage_impl.cuh and take from it what they do when a wait
// runs out (stg::hands_back, stg::drain_first, stg::full_parity).  The program reports
//   rearm     a producer's arrival on a full barrier whose phase is not the stage's, or its second on one phase
//   overlap   a copy issued into a buffer with a copy in flight
//   early     a wait for the producer's own copies at its end that returned before they had landed
//   ended     copies in flight when every agent had left
//
// usage: model_ring seed runs skip_stage limit_producer limit_consumer [plant]
//   skip_stage: stage that is never issued (-1: none); plant: consumers hand buffers back after a wait ran out
// prints: rearm overlap early ended finished (runs in which every stage was consumed) timed_out
#include <cstdio>
#include <cstdlib>
#include <random>
#include <vector>

#include "stage_impl.cuh"

using namespace rtpn::stg;

struct Barrier {
    int count = 0, arrived = 0, tx = 0, phase = 0;  // phase: the one in progress
    void settle() {
        if (arrived >= count && tx == 0) {
            ++phase;
            arrived = 0;
        }
    }
    bool done(unsigned parity) const { return ((unsigned)phase & 1u) != parity; }  // mbarrier.try_wait.parity
};

struct Copy {
    int buf, owner, stage, left;
};

struct Model {
    int nb, total, skip, limp, limc;
    bool plant;
    std::mt19937 rng;
    std::vector<Barrier> full, empty;
    std::vector<Copy> copies;
    long long rearm = 0, overlap = 0, early = 0, ended = 0;
    bool timed_out = false;
    struct Producer {
        int s = 0, polls = 0, drain = -1;
        bool out = false;
        std::vector<int> armed;  // last phase armed, by buffer
    } prod[2];
    struct Consumer {
        int s = 0, polls = 0;
        unsigned limit = 1;
        bool out = false, complete = false;
    };
    std::vector<Consumer> cons;
    int tile;  // stages of a tile

    Model(unsigned seed, int nb_, int warps, int tile_, int tiles, int skip_, int lp, int lc, bool plant_)
        : nb(nb_), total(tile_ * tiles), skip(skip_), limp(lp), limc(lc), plant(plant_), rng(seed), full(nb_), empty(nb_),
          cons(warps), tile(tile_) {
        for (auto& b : full) b.count = kProducers;
        for (auto& b : empty) b.count = warps;
        for (auto& p : prod) p.armed.assign(nb, -1);
    }
    bool in_flight(int buf, int owner) const {
        for (auto& c : copies)
            if (c.buf == buf && (owner < 0 || c.owner == owner)) return true;
        return false;
    }
    void producer(int t) {
        Producer& p = prod[t];
        if (p.drain >= 0) {  // waiting for its own copies
            if (p.drain >= p.s) {
                p.out = true;
                return;
            }
            const int q = p.drain;
            if (q != skip) {
                const bool ok = full[q % nb].done(full_parity(q, nb));
                if (!ok && ++p.polls < limp) return;
                if (ok)
                    for (auto& c : copies)
                        if (c.owner == t && c.stage == q) ++early;
            }
            p.polls = 0;
            ++p.drain;
            return;
        }
        if (p.s == total) {
            p.drain = drain_first(p.s, nb);
            return;
        }
        const int b = p.s % nb;
        if (p.s >= nb && !empty[b].done((unsigned)(p.s / nb - 1) & 1u)) {
            if (++p.polls < limp) return;
            timed_out = true;
            p.polls = 0;
            p.drain = drain_first(p.s, nb);
            return;
        }
        p.polls = 0;
        if (p.s != skip) {
            if (full[b].phase != p.s / nb || p.armed[b] == full[b].phase) ++rearm;
            if (in_flight(b, t)) ++overlap;
            p.armed[b] = full[b].phase;
            ++full[b].arrived;
            const int n = 1 + (int)(rng() % 3);
            for (int k = 0; k < n; ++k) {
                copies.push_back({b, t, p.s, 1 + (int)(rng() % 60)});
                ++full[b].tx;
            }
            full[b].settle();
        }
        ++p.s;
    }
    void consumer(Consumer& c) {
        if (c.s == total || (c.s % tile == 0 && c.s > 0 && c.limit == 0)) {  // no tile left, or it leaves after its tile
            c.complete = c.limit != 0;
            c.out = true;
            return;
        }
        const int b = c.s % nb;
        if (c.limit != 0 && !full[b].done(full_parity(c.s, nb))) {
            if (++c.polls < limc) return;
            timed_out = true;
            c.limit = 0;
        }
        c.polls = 0;
        if (plant || hands_back(c.limit)) {
            ++empty[b].arrived;
            empty[b].settle();
        }
        ++c.s;
    }
    bool run() {
        const int agents = kProducers + (int)cons.size();
        for (long long step = 0; step < 4000000; ++step) {
            bool all = true;
            for (auto& p : prod) all &= p.out;
            for (auto& c : cons) all &= c.out;
            if (all) break;
            const int k = (int)(rng() % (agents + 1));
            if (k < kProducers) {
                if (!prod[k].out) producer(k);
            } else if (k < agents) {
                if (!cons[k - kProducers].out) consumer(cons[k - kProducers]);
            }
            for (size_t i = 0; i < copies.size();) {
                if (--copies[i].left > 0) {
                    ++i;
                    continue;
                }
                Barrier& f = full[copies[i].buf];
                --f.tx;
                copies[i] = copies.back();
                copies.pop_back();
                f.settle();
            }
        }
        for (auto& p : prod)
            if (!p.out) return false;
        for (auto& c : cons)
            if (!c.out) return false;
        ended += (long long)copies.size();
        return true;
    }
};

int main(int argc, char** argv) {
    if (argc < 6) return 2;
    const unsigned seed = (unsigned)atoi(argv[1]);
    const int runs = atoi(argv[2]), skip = atoi(argv[3]), lp = atoi(argv[4]), lc = atoi(argv[5]);
    const bool plant = argc > 6;
    long long rearm = 0, overlap = 0, early = 0, ended = 0, finished = 0, timed = 0;
    for (int r = 0; r < runs; ++r) {
        std::mt19937 g(seed * 7919u + r);
        const int nb = 2 + (int)(g() % 7), tile = nb + 2 + (int)(g() % 20);
        Model m(seed + 31u * r, nb, 1 + (int)(g() % 6), tile, 1 + (int)(g() % 4), skip, lp, lc, plant);
        if (!m.run()) {
            fprintf(stderr, "an agent never left\n");
            return 3;
        }
        rearm += m.rearm;
        overlap += m.overlap;
        early += m.early;
        ended += m.ended;
        timed += m.timed_out;
        bool fin = true;
        for (auto& c : m.cons) fin &= c.complete;
        finished += fin;
    }
    printf("%lld %lld %lld %lld %lld %lld\n", rearm, overlap, early, ended, finished, timed);
    return 0;
}
