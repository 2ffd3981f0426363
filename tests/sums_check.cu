// Host check of the sums that the FP32 kernels use (csrc/common.cuh): errors of a norm's sum of
// squares over 608 threads of `rows` rows each, relative to the exact one, by
//   folded: SquareSums per thread, pairs across threads (the library's form);
//   plain:  one FP32 accumulator per thread over at most 108 rows, FP64 across threads;
//   pairs / doubles: the folded threads' sums across threads as pairs and in FP64.
// Prints: rows, RMS error folded, RMS error plain, largest |pairs - doubles| / sum.
#include <cmath>
#include <cstdio>
#include <random>
#include <vector>

#include "common.cuh"

int main() {
    const int blocks = 76, per_block = 8, trials = 96;   // as the library's grids: rows of a block, then blocks
    for (int rows : {1, 63, 64, 65, 216, 862}) {
        std::mt19937_64 gen(7);
        std::normal_distribution<double> normal(0.0, 1.0);
        double folded = 0, plain = 0, split = 0;
        for (int t = 0; t < trials; ++t) {
            long double exact = 0;
            double fp64 = 0, across = 0;
            mg::PairF pairs, block;
            for (int k = 0; k < blocks * per_block; ++k) {
                mg::SquareSums<float, 1> s;
                float acc = 0;
                for (int i = 0; i < rows; ++i) {
                    const float x = (float)normal(gen), y = (float)normal(gen);
                    exact += (long double)x * x + (long double)y * y;
                    s.add(0, x, y);
                    s.end_row();
                    acc = std::fma(x, x, std::fma(y, y, acc));
                    if (i % 108 == 107 || i + 1 == rows) {
                        fp64 += acc;
                        acc = 0;
                    }
                }
                s.fold();
                block.add(s.total[0]);
                if (k % per_block + 1 == per_block) {
                    pairs.add(block);
                    block = mg::PairF();
                }
                across += s.total[0].value();
            }
            folded += std::pow((double)((pairs.value() - exact) / exact), 2);
            plain += std::pow((double)((fp64 - exact) / exact), 2);
            split = std::fmax(split, std::fabs(pairs.value() - across) / across);
        }
        std::printf("%d %.6e %.6e %.6e\n", rows, std::sqrt(folded / trials), std::sqrt(plain / trials), split);
    }
}
