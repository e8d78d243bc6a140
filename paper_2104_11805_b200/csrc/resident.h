// Plan of the kernel that keeps a whole network's activations in shared memory (resident.cuh): which nets and batches it takes, how
// its memory is cut, and in which order the entries of eight rows are read.  Plain code, so that it can be looked at without a device.
#pragma once
#include <stdint.h>

#include <algorithm>

#ifdef __CUDACC__
#define SDNN_HD __host__ __device__ __forceinline__
#else
#define SDNN_HD inline
#endif

namespace sdnn_plan {

constexpr int RES_UNIT = 32;              // rows of a unit: one per lane of a warp
constexpr int RES_CLASSES = 8;            // 16-byte columns of shared memory: slots s and t meet in a bank where s = t modulo 8
constexpr int RES_WARPS = 16;
constexpr int RES_BLOCK = 1024;           // rows among which groups of eight are chosen
constexpr int RES_MAX_ROW = 248;          // entries of a row: counts and places are kept in bytes
constexpr int RES_SMEM = 226 * 1024;

// One step of a group of eight rows, of `left` that are left: which class each row reads from.  have: byte c = mask of the rows that
// still have an entry of class c; total[c]: entries of class c that the group still has; must: rows that have to read now (no step to
// spare).  Returns a class per row, four bits each, 15 = the row waits.
// While no class has more entries than there are steps, the rows read eight different ones (the rest can then always be read that
// way: a bipartite graph of rows and classes falls apart into as many matchings as its largest degree).  Else one or more classes have
// to be read twice in some step, which costs that step a second wavefront whatever else is read twice in it: so this step reads
// as many entries twice as bring the classes to the number of steps that will be left.  With rows of equal length the steps
// that take two wavefronts are as few as the group's counts allow: the largest distance of a class from the mean.
// A largest matching of classes (twice: and of second copies of classes) with rows by augmenting paths, the fullest classes first.
SDNN_HD uint32_t resident_step(uint64_t have, const int (&total)[RES_CLASSES], uint32_t must, int left) {
    int key[RES_CLASSES];
    for (int c = 0; c < RES_CLASSES; ++c) key[c] = total[c] * RES_CLASSES + c;
#define SDNN_ORDER(A, B) { const int hi_ = key[A] > key[B] ? key[A] : key[B], lo_ = key[A] > key[B] ? key[B] : key[A]; key[A] = hi_; key[B] = lo_; }
    SDNN_ORDER(0, 2) SDNN_ORDER(1, 3) SDNN_ORDER(4, 6) SDNN_ORDER(5, 7)
    SDNN_ORDER(0, 4) SDNN_ORDER(1, 5) SDNN_ORDER(2, 6) SDNN_ORDER(3, 7)
    SDNN_ORDER(0, 1) SDNN_ORDER(2, 3) SDNN_ORDER(4, 5) SDNN_ORDER(6, 7)
    SDNN_ORDER(2, 4) SDNN_ORDER(3, 5)
    SDNN_ORDER(1, 4) SDNN_ORDER(3, 6)
    SDNN_ORDER(1, 2) SDNN_ORDER(3, 4) SDNN_ORDER(5, 6)
#undef SDNN_ORDER
    // nodes in the order they are matched: class, or class + 8 for the second copy
    uint64_t order = 0;
    int nodes = 0;
    const bool twice = key[0] / RES_CLASSES > left;
    for (int i = 0; i < RES_CLASSES; ++i)
        if (!twice || key[i] / RES_CLASSES >= left) order |= (uint64_t)(key[i] & 7) << (4 * nodes++);
    if (twice) {
        for (int i = 0; i < RES_CLASSES; ++i)
            if (key[i] / RES_CLASSES > left) order |= (uint64_t)((key[i] & 7) | 8) << (4 * nodes++);
        for (int i = 0; i < RES_CLASSES; ++i)
            if (key[i] / RES_CLASSES < left) order |= (uint64_t)(key[i] & 7) << (4 * nodes++);
    }
    uint64_t of_node = 0;                 // row of each matched node, node of each matched row: four bits each
    uint32_t of_row = 0, rows_set = 0, nodes_set = 0;
    for (int i = 0; i < nodes && rows_set != 0xffu; ++i) {
        uint64_t queue = (order >> (4 * i)) & 15u;
        uint32_t from = 0, seen = 0;      // node each row was reached from
        int head = 0, tail = 1, end = -1;
        while (head < tail && end < 0) {
            const uint32_t q = (uint32_t)(queue >> (4 * head++)) & 15u;
            uint32_t rows = (uint32_t)(have >> (8 * (q & 7u))) & 0xffu & ~seen;
            for (int r = 0; r < RES_CLASSES && rows >> r; ++r) {
                if (!((rows >> r) & 1u)) continue;
                seen |= 1u << r;
                from = (from & ~(15u << (4 * r))) | q << (4 * r);
                if (!((rows_set >> r) & 1u)) { end = r; break; }
                queue |= (uint64_t)((of_row >> (4 * r)) & 15u) << (4 * tail++);
            }
        }
        if (end < 0) continue;
        rows_set |= 1u << end;
        for (int r = end;;) {             // hand the rows of the path on to the node each was reached from
            const uint32_t q = (from >> (4 * r)) & 15u;
            const bool had = (nodes_set >> q) & 1u;
            const int before = (int)((of_node >> (4 * q)) & 15u);
            of_row = (of_row & ~(15u << (4 * r))) | q << (4 * r);
            of_node = (of_node & ~((uint64_t)15u << (4 * q))) | (uint64_t)r << (4 * q);
            nodes_set |= 1u << q;
            if (!had) break;
            r = before;
        }
    }
    uint32_t read = 0, load = 0;          // class of each row; rows reading each class, four bits each
    for (int r = 0; r < RES_CLASSES; ++r) {
        const uint32_t c = (of_row >> (4 * r)) & 7u;
        if ((rows_set >> r) & 1u) { read |= c << (4 * r); load += 1u << (4 * c); }
        else read |= 15u << (4 * r);
    }
    for (int r = 0; r < RES_CLASSES; ++r) {      // rows of different lengths: one may be left over that cannot wait
        if (!((must >> r) & 1u) || ((rows_set >> r) & 1u)) continue;
        int best = -1, best_key = 0;
        for (int c = 0; c < RES_CLASSES; ++c) {
            if (!((have >> (8 * c + r)) & 1u)) continue;
            const int k = (int)((load >> (4 * c)) & 15u) * 65536 - total[c];
            if (best < 0 || k < best_key) { best = c; best_key = k; }
        }
        if (best >= 0) {
            read = (read & ~(15u << (4 * r))) | (uint32_t)best << (4 * r);
            load += 1u << (4 * best);
        }
    }
    return read;
}

// Class of the zeros that a waiting row reads: the rows that wait share out the classes that nobody reads.
SDNN_HD int resident_idle_class(uint32_t of_row, int row) {
    uint32_t read = 0;
    int before = 0;
    for (int r = 0; r < RES_CLASSES; ++r) {
        const uint32_t c = (of_row >> (4 * r)) & 15u;
        if (c != 15u) read |= 1u << c;
        else if (r < row) ++before;
    }
    for (int c = 0; c < RES_CLASSES; ++c)
        if (!((read >> c) & 1u) && before-- == 0) return c;
    return 0;
}

// How the kernel holds a net of n neurons with 4 p inputs to a CTA.  A layer's activations are `slots` slots of 16 p bytes; outputs go
// to the free slots of a ring of `cap`, and what does not fit stays in the registers of the warps' last `held` units until the
// layer has been read.  ok = false: it does not fit at all.
struct ResidentShape { bool ok; int units, slots, cap, held; };
SDNN_HD ResidentShape resident_shape(int n, int p) {
    ResidentShape s{};
    s.units = (n + RES_UNIT - 1) / RES_UNIT;
    s.slots = s.units * RES_UNIT + RES_CLASSES;      // the last eight hold zeros, one of each class
    const int fit = RES_SMEM / (16 * p) / RES_CLASSES * RES_CLASSES, rounds = (s.units + RES_WARPS - 1) / RES_WARPS;
    if (2 * s.slots <= fit) { s.ok = true; s.cap = 2 * s.slots; return s; }
    if (s.slots > fit) return s;
    s.cap = fit;
    const int free_rounds = (fit - s.slots) / RES_UNIT / RES_WARPS, most = p <= 2 ? 4 : 2;      // registers: 4 p numbers a held unit
    s.held = rounds - free_rounds <= 2 ? 2 : 4;
    s.ok = rounds - free_rounds <= most && rounds >= s.held;
    return s;
}

// How a batch is cut into CTAs.  Rounds of 4 p inputs on every SM as long as they are whole; what is left, less than a round, is one more
// round of CTAs that take as few inputs as that needs: the launch of each width q <= p looks whether the rest is its own.
// Where the number of inputs is known only on the device, all these launches are made, and all but one find nothing.
SDNN_HD int resident_rest_width(int rest, int sms) { return rest ? (rest + 4 * sms - 1) / (4 * sms) : 0; }
// inputs [begin, end) of `total` that the launch of width q takes
SDNN_HD void resident_share(int total, int sms, int p, int q, int* begin, int* end) {
    const int main = total / (4 * p * sms) * (4 * p * sms), rest = total - main;
    const bool own = resident_rest_width(rest, sms) == q;
    *begin = q == p ? 0 : main;
    *end = own ? total : q == p ? main : *begin;
}
// A layer: neurons, stored elements (padding included), entries of the longest row, whether rows differ in length.
struct ResidentLayer { int n; double elems; int longest; bool several; };
// What a layer takes, in clocks, one way and the other, fitted to measurements of both (24 layers of 600 .. 8000 neurons, 16, 32 and 56 entries a row, 8 to 56
// and Poisson(32); us per layer, layer launches / this kernel, 32 entries):
//   neurons   256 inputs      400             592             1184            2368            4000
//     640     3.49 / 3.83     4.59 / 3.88     4.75 / 3.90     7.71 / 5.22     13.5 / 8.2      18.7 / 14.8
//    1024     3.50 / 4.75     4.72 / 4.75     6.85 / 4.79     9.52 / 6.84     18.5 / 11.4     27.2 / 20.5
//    2048     4.86 / 8.35     7.96 / 8.39     11.0 / 8.45     17.3 / 12.7     34.9 / 22.3     54.0 / 39.6
//    4096     8.75 / 15.5     17.4 / 15.5     19.9 / 15.6     33.4 / 24.9     67.0 / 50.0     109 / 90.7
//    8000     17.0 / 33.2     27.1 / 33.8     38.4 / 34.7     66.2 / 70.4     131 / 134
// A round of CTAs: wavefronts of operands (1.06 for eight of them), entries (6 bytes each) and outputs.  Units held in registers cost addresses, warps
// without a unit in the last round idle; at 4 inputs a CTA a warp waits for its entries, more so where rows differ in length (their chunks
// come in no fours; 7000 neurons, 8 to 56 entries, 592 inputs: 33.9 us, 32 each: 27.5) and where a layer of them is large.
inline double resident_clocks(const ResidentLayer& l, int p) {
    const ResidentShape s = resident_shape(l.n, p);
    const double idle = (double)((s.units + RES_WARPS - 1) / RES_WARPS * RES_WARPS) / s.units - 1;
    const double pipe = (l.elems * (p * 1.06 / 8 + 6.0 / 128) + l.n * p / 4.0) * (s.held == 4 ? 1.10 : s.held ? 1.04 : 1.0);
    const double wait = p == 1 ? 1.20 + 0.45 * idle + (l.several ? 0.13 : 0.0) + 0.056e-5 * std::max(0.0, l.elems - 130000)
                               : 1.03 + 0.035 * (p - 1) + (p == 2 ? 0.20 : 0.165) * idle + (l.several ? 0.02 : 0.0);
    return pipe * wait + 2400;
}
// ... for `inputs` inputs in rounds of width p; a rest behind whole rounds finds the CTAs out of step, which then read other parts of the network
// (5000 neurons, 16 entries, 1500 and 1776 inputs: 38 and 34 us a layer)
inline double resident_clocks(const ResidentLayer& l, int64_t inputs, int sms, int p) {
    const int64_t round = (int64_t)4 * p * sms;
    const int q = resident_rest_width((int)(inputs % round), sms);
    const double whole = (double)(inputs / round) * resident_clocks(l, p);
    return (whole + (q ? resident_clocks(l, q) : 0.0)) * (whole > 0 && q ? (p == 1 ? 1.08 : 1.03) : 1.0);
}
// The layer launches, in tiles of `tile` inputs: 66 bytes of operands per clock and SM (some of which L1 has: 80 for a row's entries, which its end takes a part of), and the round trips of
// the longest row, which a second tile in flight fills in part.  A small batch pays for a part of the padding to whole chunks of 256.
inline double launch_clocks(const ResidentLayer& l, int64_t inputs, int sms, int tile) {
    const double trips = 4640 + 177.0 * l.longest;
    const double padded = (double)inputs + (inputs <= tile && l.elems * (double)inputs < (32 << 20) ? 0.3 * (double)((256 - inputs % 256) % 256) : 0.0);
    const double gathers = (0.82 * l.elems + 7.5 * l.n) * padded * 4.0 / (66.0 * sms);
    const double tiles = (double)((inputs + tile - 1) / tile);
    return inputs <= tile ? std::max(trips, gathers + 0.48 * trips) : std::max(0.66 * tiles * trips, gathers + 0.19 * tiles * trips);
}
// ... dropping dead inputs, where `inputs` of those in all tiles are left
inline double dropping_clocks(const ResidentLayer& l, int64_t inputs, int sms, int tiles) {
    const double trips = 4640 + 177.0 * l.longest, gathers = (0.82 * l.elems + 7.5 * l.n) * (double)inputs * 4.0 / (66.0 * sms);
    return tiles == 1 ? 1.5 * gathers + 0.85 * trips + 1800 : 1.25 * gathers + 0.5 * tiles * trips + 1500;
}
// The width for `inputs` inputs, 0 where the layer launches, in tiles of `tile` inputs, are faster.  drop: dead inputs are dropped.  How many are left
// after a few layers is not known: a third decides between the two ways, and the width is one that is right for a third and for all of them.
inline int resident_width(const ResidentLayer& l, int64_t inputs, int sms, int tile, bool drop) {
    int best = 0;
    if (inputs <= 256) return best;      // a single chunk of inputs: the table's first column
    double least = launch_clocks(l, inputs, sms, tile);
    for (int p = 1; p <= 4 && resident_shape(l.n, p).ok; ++p) {      // where a width does not fit, nor does a wider one
        const double all = resident_clocks(l, inputs, sms, p);
        if (all < least) { least = all; best = p; }
    }
    if (!drop || !best) return best;
    const int64_t third = (inputs + 2) / 3;
    auto either = [&](int p) { return resident_clocks(l, inputs, sms, p) + 3 * resident_clocks(l, third, sms, p); };
    for (int p = 1; p <= 4 && resident_shape(l.n, p).ok; ++p) if (either(p) < either(best)) best = p;
    return resident_clocks(l, third, sms, best) < dropping_clocks(l, third, sms, (int)((inputs + tile - 1) / tile)) ? best : 0;
}
inline int resident_width(int n, double elems, int64_t inputs, int sms, int tile, bool drop) {      // rows of one length
    return resident_width(ResidentLayer{n, elems, (int)(elems / n), false}, inputs, sms, tile, drop);
}

// A batch from host memory that is one tile goes in two pieces, so that one's copies run under the other's layers.  Halves of 4 inputs a
// CTA whose CTAs fit the device together cost no round of their own (us, layer launches / halves: 3000 x 40, 592 inputs 952 / 717, rows of 8 to
// 56 entries 957 / 829; 1500 x 60 738 / 521; 700 x 60, 300 inputs 344 / 292).  Not where the copies weigh as much as the layers (4096 x 40, 592
// inputs 1003 / 974 and 1082 / 1150), nor as 8 and 4 inputs a CTA beyond that (3000 x 40, 700 inputs 927 / 931, 4096 x 40, 900 1434 / 1487): there both
// halves go through the layer launches, which fill each other's gaps.  Returns the inputs of the first half, 0: not this way.
constexpr int RES_HALVES = 3072;      // most neurons
inline int resident_half(int n, int64_t inputs, int sms) {
    return n <= RES_HALVES && inputs >= 8 && (inputs + 3) / 4 <= sms ? (int)((inputs + 7) / 8) * 4 : 0;
}
// ... and only where it pays: halves of up to 256 inputs are a single chunk of the layer launches, which wider nets then go through faster (time of
// halves / of layer launches, 40 layers, equal rows: 2048 neurons, 450 inputs 1.20 (381 us in layer launches), 1800, 500 1.21, 2048, 550 0.90, 1024, 450 1.01,
// 700, 450 0.89).
inline int resident_half_pays(int n, int64_t inputs, int sms) { return inputs > 512 || n <= 1024 ? resident_half(n, inputs, sms) : 0; }

}  // namespace sdnn_plan
