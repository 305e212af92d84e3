// Index words by their number of ones.  A state of fixed electron number is zero
// wherever the index has another count, and an aligned run of 2^nb bit positions
// whose other bits are known holds the amplitudes of one class of nb-bit words.
#pragma once

#include <cstdint>

namespace vqe {

constexpr int kClassBits = 12;

// The nb-bit words in order of their number of ones, for nb = 0..kClassBits one
// after the other (nb's from 2^nb - 1), the place of every word inside its
// class of equal popcount, and where the classes begin.
struct ClassTables {
    uint16_t word[2 << kClassBits] = {}, place[2 << kClassBits] = {};
    uint16_t begin[kClassBits + 1][kClassBits + 2] = {};
    constexpr ClassTables() {
        for (int nb = 0; nb <= kClassBits; ++nb) {
            const int at = (1 << nb) - 1;
            int next[kClassBits + 1] = {}, ones = 0;
            for (int p = 0, c = 1; p <= nb; ++p) {   // c = binomial(nb, p)
                next[p] = ones;
                begin[nb][p] = uint16_t(ones);
                ones += c;
                begin[nb][p + 1] = uint16_t(ones);
                c = c * (nb - p) / (p + 1);
            }
            for (int v = 0; v < (1 << nb); ++v) {
                int pc = 0;
                for (int t = v; t; t &= t - 1) ++pc;
                place[at + v] = uint16_t(next[pc] - begin[nb][pc]);
                word[at + next[pc]++] = uint16_t(v);
            }
        }
    }
};
__device__ constexpr ClassTables kClass{};

}  // namespace vqe
