// Host model of the sums over CTAs of a persistent kernel (csrc/cta_sums.cuh):
// every CTA stores its part of a sum, meets the others at a barrier and reads all
// parts.  Between two barriers the CTAs run in any order, so at every sum one CTA
// (each in turn) is held back: it reads only when all others have stored their
// parts of the next sum and stand at its barrier.
#include <cstdio>
#include <vector>

#include "cta_sums.cuh"

int main() {
    const int ctas = 5, sums = 9;
    for (int late = 0; late < ctas; ++late) {
        std::vector<float> part(lace::CtaSums::kRows * ctas, -1.f);
        std::vector<lace::CtaSums> s(ctas);
        auto store = [&](int c, int t) { part[s[c].at(c, ctas)] = (float)(100 * t + c); };
        auto read = [&](int c, int t) {
            for (int b = 0; b < ctas; ++b)
                if (part[s[c].at(b, ctas)] != (float)(100 * t + b)) {
                    std::printf("sum %d: CTA %d reads %g for CTA %d\n", t, c, (double)part[s[c].at(b, ctas)], b);
                    return false;
                }
            s[c].next();
            return true;
        };
        for (int c = 0; c < ctas; ++c) store(c, 0);
        for (int t = 0; t < sums; ++t) {  // the barrier of sum t is passed
            for (int c = 0; c < ctas; ++c) {
                if (c == late) continue;
                if (!read(c, t)) return 1;
                if (t + 1 < sums) store(c, t + 1);
            }
            if (!read(late, t)) return 1;
            if (t + 1 < sums) store(late, t + 1);
        }
    }
    std::printf("ok\n");
    return 0;
}
