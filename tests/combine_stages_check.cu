// Host model of the hand-offs of combine_ws_kernel (csrc/tc_combine.cuh): the copying
// thread, the MMA thread and two sets of cut warps that take the even and the odd
// steps, with the kernel's numbers of stages.  mbarriers know the parity of their phase
// only, as the hardware's; rows land in any order, and every thread advances at
// random.  A cut warp has to find its own step's rows in a stage, and all have to finish.
#include <cstdio>
#include <random>
#include <vector>

#include "tc_combine.cuh"

namespace {

struct Slices2 {
    static constexpr int SLICES = 2, ACCS = 1;
    static constexpr uint32_t FORMAT = 1;
};
struct Slices3 {
    static constexpr int SLICES = 3, ACCS = 3;
    static constexpr uint32_t FORMAT = 0;
};

struct Bar {
    int count, left, phase = 0;
    explicit Bar(int n = 1) : count(n), left(n) {}
    void arrive() {
        if (--left == 0) ++phase, left = count;
    }
    // what a wait for the phase of this parity sees
    bool passed(int parity) const { return (phase & 1) != parity; }
};

constexpr int kWarps = 2;  // a set (the kernel's eight, fewer for the model)

struct Model {
    int A, T, nsteps, tiles, total;
    std::mt19937& rng;
    std::vector<Bar> full, empty, cut, mma;
    Bar tile{1}, drained{2 * kWarps};
    std::vector<int> stage;
    std::vector<int> pending;  // copies in flight
    int pg = 0, mg = 0;        // steps copied, steps multiplied
    struct Warp {
        int set, t = 0, g, last, part = 0;  // part of its step; last: the tile before is written
        bool done = false;
    };
    std::vector<Warp> warps;

    Model(int a, int tst, int n, int k, std::mt19937& r)
        : A(a), T(tst), nsteps(n), tiles(k), total(n * k), rng(r), full(a, Bar(1)), empty(a, Bar(kWarps)), cut(tst, Bar(kWarps)),
          mma(tst, Bar(1)), stage(a, -1) {
        for (int w = 0; w < 2 * kWarps; ++w) {
            Warp x{w & 1};
            x.g = x.set & 1, x.last = 1;
            warps.push_back(x);
        }
    }
    bool producer() {
        if (pg >= total) return false;
        const int s = pg % A;
        if (pg >= A && !empty[s].passed((pg / A - 1) & 1)) return false;
        pending.push_back(pg++);
        return true;
    }
    bool land() {
        if (pending.empty()) return false;
        const int i = (int)(rng() % pending.size()), g = pending[i];
        pending.erase(pending.begin() + i);
        stage[g % A] = g;
        full[g % A].arrive();
        return true;
    }
    bool multiply() {
        if (mg >= total || !cut[mg % T].passed((mg / T) & 1)) return false;
        if (mg > 0 && mg % nsteps == 0 && !drained.passed((mg / nsteps - 1) & 1)) return false;
        mma[mg % T].arrive();
        if (mg % nsteps == nsteps - 1) tile.arrive();
        ++mg;
        return true;
    }
    // one move of a cut warp; *ok = false: it read another step's rows
    bool step(Warp& w, bool* ok) {
        if (w.done) return false;
        const int end = (w.t + 1) * nsteps;
        if (w.part == 0 && w.g < end) {
            if (!full[w.g % A].passed((w.g / A) & 1)) return false;
            w.part = 1;
        } else if (w.part == 1) {
            if (w.g >= T && !mma[w.g % T].passed((w.g / T - 1) & 1)) return false;
            *ok = stage[w.g % A] == w.g;
            empty[w.g % A].arrive();
            cut[w.g % T].arrive();
            w.g += 2;
            w.part = w.last ? 0 : 2;
        } else {  // the tile before (after this tile's first step, or with no step of this tile)
            if (!w.last) {
                if (!tile.passed((w.t - 1) & 1)) return false;
                drained.arrive();
                w.last = 1;
            }
            w.part = 0;
            if (w.g >= end) {
                if (++w.t == tiles) w.done = true;
                w.last = 0;
                w.g = w.t * nsteps + ((w.t * nsteps ^ w.set) & 1);
            }
        }
        return true;
    }
    const char* run() {
        for (int idle = 0; idle < 4000;) {
            bool ok = true, all = true;
            for (auto& w : warps) all &= w.done;
            if (all) return nullptr;
            const int who = (int)(rng() % (5 + warps.size()));
            const bool moved = who == 0 ? producer() : who == 1 ? (rng() % 4 == 0 && land()) : who < 5 ? multiply() : step(warps[who - 5], &ok);
            if (!ok) return "a cut warp read the rows of another step";
            idle = moved ? 0 : idle + 1;
        }
        return "nothing moves any more";
    }
};

template <class S, int NT> bool check(const char* name) {
    using C = lace::CombineShape<S, NT>;
    std::mt19937 rng(NT + S::SLICES);
    for (int k = 0; k < 4000; ++k) {
        Model m(C::ASTAGES, C::TSTAGES, 1 + (int)(rng() % 14), 2 + (int)(rng() % 4), rng);
        if (const char* e = m.run()) {
            std::printf("%s, %d stages, %d steps, %d tiles: %s\n", name, C::ASTAGES, m.nsteps, m.tiles, e);
            return false;
        }
    }
    return true;
}

}  // namespace

int main() {
    const bool ok = check<Slices2, 64>("two slices, 64") && check<Slices2, 128>("two slices, 128") &&
                    check<Slices2, 256>("two slices, 256") && check<Slices3, 128>("three slices, 128");
    if (ok) std::printf("ok\n");
    return ok ? 0 : 1;
}
