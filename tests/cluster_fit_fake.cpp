// cluster_that_fits against a fake GPU: argv: want, largest cluster that fits
// (0: none; -1: the query fails).  Prints the choice.
#include <cstdio>
#include <cstdlib>

#include "cluster_fit.cuh"

int main(int, char **argv) {
    const int want = std::atoi(argv[1]), room = std::atoi(argv[2]);
    std::printf("%d\n", img::cluster_that_fits(want, [&](int c) { return room < 0 ? -1 : c <= room ? 1 : 0; }));
}
