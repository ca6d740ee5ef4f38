// When a run takes two steps per launch (lb_pair.cuh): host code, sizes only.
#pragma once

namespace trt {

// The lattices that would share the launches of a run.
struct PairRun {
    int members;          // lattices
    long long nodes;      // in all
    long long columns;    // nodes that their strips store, lattice or not (strips x width x ny)
    long long tiled;      // G_CURRENT: nodes that the 32-wide tiles of its single steps cover
    int elem;             // bytes of a stored population, 4 or 2
    bool current, off;    // Phi at the current level, no G; else lagged
    bool general;         // walls, a mask or open edges
    bool ghosts;          // outlet ghosts, whose single steps take a second launch per lattice
    bool mask, crowded;   // a mask; at least half of the row segments near its walls
    long long padded;     // nodes with the rows' padding
    int depth;            // G_CURRENT: launches of a single step one after the other
    bool replayed;        // launches from a captured graph, not by the host one by one
    bool batch;           // launches of a batch, not of one lattice's own steps
};

// Small launches of two steps last as long as one warp's walk: a band of two rows
// takes four row collisions in a row, 3.7 us periodic and 8 us with walls (a step:
// half), whatever the lattice's size.  Single steps of few nodes are faster than
// that where the host does not bound their launches.  us per step, two steps per
// launch / single, on GB300, replayed unless stated:
//  - lagged or off, periodic: always.  64^2 1.9 / 2.6, 512^2 3.3 / 4.9 against the
//    vector kernel; against the scalar one, where nx is no multiple of the vector, 66 x
//    64 1.9 / 1.7, 190^2 1.9 / 1.9, 250 x 246 2.2 / 2.0, 330^2 2.2 / 2.6, but half the
//    launches weigh more in whole solves: 187 x 56 BF16, 32 steps launched by the host,
//    79 / 106 us, two of 70 x 90 FP16, 110 steps in a batch, 91 / 103;
//  - outlet ghosts: always faster, 64^2 5.2 / 9.0, 1024^2 19.7 / 21.3;
//  - walls, lagged: 64^2 4.1 / 2.7, 512^2 5.6 / 5.3, 768^2 8.4 / 8.9; 16 lattices of
//    64 x 1024, whose strips store 60 of their 64 columns and then 4, 19.9 / 14.9,
//    of 100 x 1024 22.6 / 31.8: nodes weighted by the square of the share of the
//    strips' columns that are in the lattice, from 400,000 on; without G 448^2
//    3.8 / 4.1: from 160,000.  Below a share of 0.6 only out of L2: FP32 24 lattices
//    of 32 x 4096 50 / 54, 16-bit 54 / 49, 90 of them 170 / 178;
//  - masks without ghosts: a few walls make whole strips slow that single steps take in
//    their stride, so only out of L2: 1024^2 with a block 14.5 / 12.7, 1280^2 20.7 / 19.9,
//    1536^2 22.1 / 37.1 (without G 512^2 4.8 / 5.1); where walls are everywhere single
//    steps are slow too, and the line is that of open walls: 5 % of solid nodes, 768^2
//    12.8 / 14.7, 40 lattices of 128^2 18.3 / 16.5;
//  - Phi at the current level: launched one by one, single steps are bound by the
//    host (64^2 3.7 / 6.1, 512^2 6.9 / 8.2); replayed, FP32 512^2 7.0 / 6.0, 640^2 8.4 /
//    8.3, 16-bit 640^2 8.6 / 7.2, 768^2 9.3 / 10.9, and 40 lattices of 64^2, which take
//    three launches one after the other, 7.1 / 11.4.
//  - launches that the host makes one by one for a batch: its kernel of single steps,
//    which looks the lattice up, takes 0.7 us longer than a lattice's own (one of 510 x
//    512 with walls FP16 5.2 / 5.2, alone 5.2 / 4.4; a whole solve of 248 x 1518 BF16, 16
//    steps, 71 / 86 us), and the arguments of more than 4 lattices (up to 26 KB a launch)
//    longer still: with walls FP32 8 lattices of 130 x 126 4.8 / 5.1, 16 of 66 x 64 4.7 /
//    3.7.
inline bool two_steps_pay(const PairRun& r) {
    if (r.current) return !r.replayed || r.depth >= 2 || r.tiled >= (r.elem == 4 ? 400000 : 500000);
    if (!r.general) return true;
    if (r.ghosts) return true;
    const double share = (double)r.nodes / (double)r.columns;
    if (!r.replayed && r.members > 4) return (double)r.nodes * share * share >= 40e3;
    if (r.mask && !r.crowded && !r.off) return r.padded >= 1900000;
    const double least = share < 0.6 ? (r.elem == 4 ? 800e3 : 3e6) : (r.off && !r.mask ? 160e3 : (r.batch && !r.replayed ? 230e3 : 400e3));
    return (double)r.nodes * share * share >= least;
}

}  // namespace trt
