// Which of the compiled kernels a batch runs: rules on its sizes, on the host.  All kernels of a
// stage write the same neighbour lists and, in the FP32 forms, the same bits.
#pragma once

#include "nep_common.cuh"

namespace nep {

// What a batch asks of the neighbour search: the distance tests of all its particles and, of the
// request whose particles have most of them, a particle's tests, the model's types and whether
// its cells are one.  Counted from the cells' mean population.
struct NeighborLoad {
    int n = 0, ncell = 0;
    double tests = 0.0, most = 0.0;
    int types = 1;
    bool one_cell = false;
    int items = 0;  // work items
    void add(const CellGrid& g, int n_r, int n_types)
    {
        double stencil = 1.0;  // cells around a particle's
        for (int a = 0; a < 3; ++a) stencil *= g.pbc[a] ? 2 * g.S[a] + 1 : (g.nc[a] < 3 ? g.nc[a] : 3);
        const double t = stencil * n_r / g.ncell;
        n += n_r;
        ncell += g.ncell;
        items += (n_r + kBlock - 1) / kBlock;
        tests += t * n_r;
        if (t > most) {
            most = t;
            types = n_types;
            one_cell = g.ncell == 1;
        }
    }
};

// The neighbour kernel of a batch: the particles that a warp takes (1 or 8), or 0 for one thread per
// particle.  A thread that tests all candidates of its particle takes the same time with
// one block on the chip as with three on every SM, and a batch ends with the particles that
// have most candidates; the warp kernels' time grows with the sum of all tests.  So the line is
// the number of particles that the tests would make if each had as many as the batch's densest
// request (that of a single configuration is its number of particles).  Measured (FP32, us;
// one warp per particle / per eight / one thread per particle):
//   water         9,200 particles 35 / 35 / 66, 11,500 47 / 45 / 72, 33,000 98 / 58 / 71,
//                 39,000 107 / 72 / 70, 58,000 152 / 86 / 78
//   two types     33,000 101 / 61 / 94, 58,000 154 / 92 / 101, 77,000 213 / 121 / 109
//   nanowire      11,500 36 / 43 / 101, 58,000 123 / 72 / 106 (three types, a dense core)
//   whole calls on batches: 100 boxes of 64 to 1,000 particles of two models, 4,000 such
//                 particles 302 / 328 / 354; boxes of 64 in one cell each, 12,800 246 / 267 / 246,
//                 19,200 309 / 298 / 266
// A thread's tests are quicker in a box of one cell, whose candidates all lanes of its warp share,
// and slower with several types (cutoffs by type pair).  Eight particles of a warp share
// little where cells hold fewer than two (a 50,000-particle monolayer, 1.2 to a cell: 73 / 36 /
// 25).  FP64 tests every pair in FP64 in the warp kernels and screens in FP32 in the
// other (water at 11,500 particles 205 / 212 / 197, a nanowire 134 / 167 / 209).
inline int neighbor_form(const NeighborLoad& w, bool fp64)
{
    if (fp64) return w.items <= 90 ? 1 : 0;
    const double particles = w.tests / w.most;
    if (particles <= 11520.0) return 1;
    if (w.n < 2 * (double)w.ncell) return 0;
    const double line = w.types > 1 ? 66000.0 : 34000.0;
    return particles <= (w.one_cell ? line / 3.0 : line) ? 8 : 0;
}

// What decides between the evaluation kernels: the batch's particles and work items (capacities),
// the models' most types, widest hidden layer and largest tables, the list capacities, and
// whether per-particle virials are returned.
struct EvalLoad {
    int n, items, types, hidden, mnR, mnA;
    size_t table_bytes;
    bool virial;
};

// Which FP32 batches run the group kernels (evaluate_group.cu).  Theirs is the shorter latency, the
// thread-per-particle kernels' the fewer instructions.  The latter take one block's time until
// every SM has one (152 work items), a little more until every SM has three (456), then
// a second wave's; the former grow with the particles from one wave of their blocks on (76
// full items).  Where they cross depends on a thread's serial work: with many pairs a
// particle (judged by the list capacities, about half as many again as the counts) or several
// types (whose threads wait for a neighbour's type before its gradient vector) the group
// kernels win for longer; a wide hidden layer, whose weights they read through L1, takes that
// away.  Both kernels together, us (thread / group):
//                         8,200 particles   10,200   12,300   16,400   20,500   25,600
//   water                    73 / 53         73 / 68  75 / 76  74 / 83  84 / 102 86 / 109
//   monolayer, 4 types       60 / 45         62 / 60  61 / 65  61 / 66  68 / 78  72 / 87
//   water, 300 units         128 / 98       128 / 153
//   nanowire, 3 types        111 / 59       112 / 62 113 / 82 113 / 93 114 / 100 130 / 125
//   two types                110 / 63       109 / 82 112 / 92 112 / 98 128 / 123 132 / 134
//   8 types                  123 / 76       126 / 95 125 / 107 126 / 121 159 / 147 162 / 172
//   water, r_c 12 and 8 A    166 / 92       170 / 135 169 / 142 174 / 157 210 / 205 216 / 224
// With per-particle virials a thread also scatters nine sums a pair (whole calls: water 18,400
// particles 177 / 177, monolayer 20,500 151 / 152, two types of r_c 6 A 22,500 188 / 177 and
// 30,700 201 / 214).  Tables of more than half an SM's shared memory leave it one block, so that
// the thread kernels' time doubles with the 153rd item (700 units, whole calls: 19,500
// particles 354 / 396, 20,500 596 / 523, 25,600 609 / 535).
// FP64 always runs the group kernels: bound by the FP64 pipe, they evaluate each ordered
// angular pair once and do not spill (100,000-bead water 5.01 ms; one thread per particle
// and both directions of each pair took 7.00 ms).
inline bool evaluate_by_groups(const EvalLoad& w, bool fp64)
{
    if (fp64) return true;
    const bool wide = w.hidden > 128;
    const bool many_pairs = !wide && (w.mnA >= 96 || (w.types > 1 && w.mnR >= 96));
    const int more = w.items > 456 ? 3 : w.items > 152 ? 1 : 0;  // beyond one and beyond three blocks per SM
    int line = many_pairs ? 21504 : wide ? 9728 : w.types > 1 ? 12288 : 10240;
    if (w.virial && !many_pairs && !wide) line += w.types > 1 && w.mnR >= 48 ? 10240 : 6144;
    line += 4096 * more;
    if (w.table_bytes > 113 * 1024 && more > 0) line = line > 25600 ? line : 25600;
    return w.n <= line;
}

}  // namespace nep
