// Host-side check of row_key (agatha_dev.cuh): 1024 times a cell's score over the
// whole range of scores and drifts, built with the undefined-behaviour sanitizer
// (a product of drifting values passes 2^31).  Runs on the CPU only.
#include <cstdio>

#include "agatha_dev.cuh"

int main() {
    long bad = 0, n = 0;
    for (long z = 0; z < (1L << 28); z = z < 100 ? z + 7 : z + z / 3)
        for (long score = 0; score < (1L << 20); score = score < 50 ? score + 1 : score + score / 5, ++n)
            bad += agatha::row_key((int)(score + z), 0u - (unsigned)z * 1024u) != score * 1024;
    std::printf("%ld keys, %ld wrong\n", n, bad);
    return bad != 0;
}
