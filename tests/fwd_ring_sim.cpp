// The streamed forward's hand-back protocol under commits that arrive in any
// order.  argv: barriers (0: the product's rule), stages, tasks per stage,
// seed.  Prints "ok", "early" (a warp wrote into a buffer that the MMAs of its
// last stage may still read) or "stuck".
#include <cstdio>
#include <cstdlib>
#include <random>
#include <vector>

#include "fwd_ring.cuh"

namespace R = img::fwd_ring;

int main(int argc, char **argv) {
    const int slots = std::atoi(argv[1]), stages = std::atoi(argv[2]), ntask = std::atoi(argv[3]);
    std::mt19937 rng(std::atoi(argv[4]));
    auto slot = [&](int t) { return slots ? t % slots : R::slot(t); };
    auto parity = [&](int t) { return slots ? (unsigned)(t / slots) & 1u : R::parity(t); };
    const int np = R::warps(ntask);
    std::vector<int> next(np), written(stages, 0), done(16, 0);   // done: completions per barrier
    std::vector<bool> arrived(stages, false);
    for (int w = 0; w < np; ++w) next[w] = w;
    int issued = 0;
    // completion of a parity seen by a waiter: the barrier is past it, or
    // (falsely) two phases short of it
    auto passes = [&](int t) { return ((unsigned)done[slot(t)] & 1u) != parity(t); };
    for (;;) {
        struct Move { int kind, i; };
        std::vector<Move> moves;
        bool work = false;
        for (int w = 0; w < np; ++w) {
            if (next[w] >= stages * ntask) continue;
            work = true;
            const int t = next[w] / ntask;
            if (t < 2 || passes(t - 2)) moves.push_back({0, w});
        }
        if (issued < stages) {
            work = true;
            if (written[issued] == ntask) moves.push_back({1, 0});
        }
        for (int t = 0; t < issued; ++t)
            if (!arrived[t]) moves.push_back({2, t}), work = true;
        if (!work) break;
        if (moves.empty()) return std::puts("stuck"), 0;
        const Move m = moves[rng() % moves.size()];
        if (m.kind == 0) {
            const int t = next[m.i] / ntask;
            if (t >= 2 && !arrived[t - 2]) return std::puts("early"), 0;
            ++written[t];
            next[m.i] += np;
        } else if (m.kind == 1) {
            ++issued;
        } else {
            arrived[m.i] = true;
            ++done[slot(m.i)];
        }
    }
    return std::puts("ok"), 0;
}
