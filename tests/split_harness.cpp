// split_harness.cpp -- prints the segment size that the split products take for a reaction table
// (csrc/split_layout.h, compiled for the host): order ks kt kmax T w hS hT H.
#include <cstdio>
#include <cstdlib>

#include "split_layout.h"

int main(int argc, char** argv) {
    if (argc != 10) return 2;
    double v[8];
    for (int i = 0; i < 8; ++i) v[i] = std::atof(argv[2 + i]);
    const double g = lfmm::split_growth(v[0], v[1], v[2], v[3], v[4], v[5], v[6], v[7]);
    std::printf("%d\n", lfmm::split_size(std::atoi(argv[1]), g > SP_GROWTH));
    return 0;
}
