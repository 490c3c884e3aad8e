// Where the CTAs of a persistent kernel keep their parts of a sum over all CTAs.
#pragma once

namespace lace {

// Every CTA stores its part of sum t, all meet at a grid barrier, every CTA reads
// all parts.  A CTA that has read them goes on, and stores its part of the next sum
// while others may still read: consecutive sums take the two rows by turns.  The row of
// sum t is written again for sum t + 2, after the barrier of sum t + 1, where a CTA
// arrives only once it has read sum t, whatever the path between the two sums.
struct CtaSums {
    static constexpr int kRows = 2;
    unsigned turn = 0;
    // place of a CTA's part in kRows rows of `width`
    __host__ __device__ int at(int cta, int width) const { return (int)(turn % kRows) * width + cta; }
    __host__ __device__ void next() { ++turn; }
};

}  // namespace lace
