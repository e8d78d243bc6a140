// Rules of the launches that need no device: plain host code, so that they can be looked at without one.
#pragma once
#include <stdint.h>

#include <algorithm>
#include <vector>

namespace sdnn_plan {

// padded batch width: 4, 8, .., 256, then multiples of 256
inline int padded_width(int b) {
    if (b <= 4) return 4;
    if (b <= 256) { int w = 4; while (w < b) w <<= 1; return w; }
    return (b + 255) / 256 * 256;
}

// How the columns of an inference tile of `cnt` inputs are padded and cut: chunks of cw inputs, cols of them in all.  One chunk up
// to 256 inputs and chunks of 256 beyond, unless chunks of 128 or 64 save more padding than the 5 or 10 % they may cost, in
// layers that are bound by their gathers: 4096 neurons, 300 inputs are 320 columns, not 512 (960 -> 681 us for 60 layers),
// 16384 neurons, 150 inputs 192, not 256 (631 -> 434 us for 20).  Smaller layers are bound by their chain of round trips, which
// padding does not lengthen and more chunks do (1024 neurons, 300 inputs: 517 -> 555 us for 120).
// elems: stored elements of a layer, in the mean over the net.  windows: every layer has its operands in shared memory, in chunks of
// 32 inputs or of 16, 8 or 4: whole chunks are all the padding it needs.
constexpr int64_t SHAPE_WORK = 32 << 20;      // stored elements x inputs per layer
struct TileShape { int cw, cols; };
// ls: see split_rows; a tile whose rows are shared is of whole lanes, which hold 8 inputs (the last tile of a call may have fewer).
inline TileShape tile_shape(int cnt, int64_t elems, bool windows, int ls = 0) {
    TileShape best{std::min(padded_width(cnt), 256), padded_width(cnt)};
    if (ls && best.cols < 8) best = {8, 8};
    if (windows) return cnt <= 32 ? best : TileShape{32, (cnt + 31) / 32 * 32};
    if (cnt <= 64 || elems * cnt < SHAPE_WORK) return best;
    double least = best.cols;
    for (int cw = 128; cw >= 64; cw /= 2) {
        const int cols = (cnt + cw - 1) / cw * cw;
        const double work = cols * (cw == 64 ? 1.10 : 1.05);
        if (work < least) { least = work; best = {cw, cols}; }
    }
    return best;
}

// Whether a tile's layers are launched as a graph from a handle's second call on: one launch of the host's instead of one per
// layer, which take 2.2 us each and which a layer of a narrow net does not outlast (1024 neurons x 120 layers, 256 inputs, three
// handles in turn: 300 us a call of launches).  The first call launches directly, so that a net that is asked once does not pay for
// the graph.  Layers that outlast their launch calls several times over are launched directly (4096 neurons, tiles of 1024: 27
// us a layer, 1 % slower as graphs on two streams), unless dead inputs are being dropped (track): nobody knows what is left of those.
// elems as above, whatever the layout of the layers.
constexpr int64_t GRAPH_WORK = 32 << 20;      // stored elements x columns per layer: about 7 us
inline bool tile_as_graph(int layers, int64_t elems, int cols, bool track) { return layers >= 4 && (track || elems * cols <= GRAPH_WORK); }

// Which of the `n` graphs that a lane keeps a tile takes.  `used` columns of its `cols` hold inputs (rounded up to a lane's eight: the
// launches gather no padding beyond those), and a graph made for more of them serves fewer, for the price of their padding.  A graph
// of its own, then, while there is room (4096 neurons x 60, 72 of 128 columns: 204 -> 189 us, 100 of them 197); else the narrowest that serves; else
// the one not asked for longest makes room for one that serves any tile of this shape.  So batches that vary at will make a lane
// fill its places, and after that one graph per shape (as long as there are no more shapes than places).
// Returns the place; `make` is set where the graph has to be made first, with want.used columns (which may have been raised).
struct GraphKey { int cw = 0, cols = 0, used = 0, pdl = 0, ls = 0; bool track = false, other = false; };      // ls: see split_rows; other: of the reordered copies
inline int pick_graph(const GraphKey* have, const int64_t* asked, int n, GraphKey& want, bool& make) {      // asked[q] = 0: empty
    int room = -1, serves = -1, oldest = 0;
    make = false;
    for (int q = 0; q < n; ++q) {
        if (!asked[q]) { if (room < 0) room = q; continue; }
        const GraphKey& g = have[q];
        if (g.cw == want.cw && g.cols == want.cols && g.pdl == want.pdl && g.ls == want.ls && g.track == want.track && g.other == want.other && g.used >= want.used) {
            if (g.used == want.used) return q;
            if (serves < 0 || g.used < have[serves].used) serves = q;
        }
        if (asked[q] < asked[oldest]) oldest = q;
    }
    if (room < 0 && serves >= 0) return serves;
    make = true;
    if (room >= 0) return room;
    want.used = want.cols;
    return oldest;
}

// Whole networks in one launch (vector.cuh): CTAs of the cluster, and rows a CTA works on at once; CTA r has the rows r * VECTOR_BLOCK
// .. of every VECTOR_CTAS * VECTOR_BLOCK.
constexpr int VECTOR_CTAS = 16, VECTOR_BLOCK = 64;
// CTAs that have rows of a net of n neurons.  Only these exchange activations: see vector.cuh.
constexpr int vector_ctas(int n) { return n > (VECTOR_CTAS - 1) * VECTOR_BLOCK ? VECTOR_CTAS : (n + VECTOR_BLOCK - 1) / VECTOR_BLOCK; }

// Rows gathered per us: 0.72, 0.57, 0.31 and 0.15 rows of up to 64, 128, 256 and 512 bytes per clock and SM
inline double gathers_per_us(int row_bytes, int sms) { return (row_bytes <= 64 ? 0.72 : row_bytes <= 128 ? 0.57 : row_bytes <= 256 ? 0.31 : 0.15) * 1900.0 * sms; }

// Inference: log2 of the groups of lanes that share a row, the same for every row: as many as leave no more units than 2048 warps, the
// device's fill, and no more than a row has steps of 8 entries in the mean; none where a layer's gathers take long beside the round
// trips of a row (0.77 us a step).  A function of the net and the chunk of a call's whole tiles (call_rows) alone, so that
// the kernels that drop dead inputs, in narrower chunks, add up in the same order, and so does the call's last, narrower tile.  us a layer, one group / this: 700 neurons of 32 entries,
// 6 inputs 3.63 / 2.26, 50 inputs 3.20 / 2.18, 100 inputs 3.22 / 2.62; 3000, 12 inputs 3.88 / 2.60, 50 inputs 3.80 / 3.46; 6000, 12 inputs 4.06 / 3.65;
// left alone: 6000, 28 inputs, rows of 8 to 56 entries 5.34 / 5.46; 16384, 12 inputs 4.91 / 4.99; 30000, 6 inputs 6.79 / 7.04.
inline int split_rows(int n, int64_t elems, int cw, int sms) {
    int ls = 0;
    if (cw < 8 || cw > 128 || 2.6 * elems / gathers_per_us(4 * cw, sms) > 0.77 * elems / (8.0 * n)) return 0;
    const int lanes = cw / 8;      // of a group
    while ((lanes << (ls + 1)) <= 32 && (((int64_t)n * lanes) << (ls + 1)) <= 2048 * 32 && (int64_t)n * 8 << (ls + 1) <= elems) ++ls;
    return ls;
}
// ... of all tiles of a call whose whole tiles have `tile` inputs; none where those are of several chunks
inline int call_rows(int n, int64_t elems, int tile, int sms) {
    const TileShape whole = tile_shape(tile, elems, false);
    return whole.cw == whole.cols ? split_rows(n, elems, whole.cw, sms) : 0;
}

// Allocation-free calls: groups of lanes that share a row of the caller's CSR arrays (at least so many), and whether a single group is of lanes of 4
// inputs instead of 8 (`narrow`).  width: inputs of a chunk; per_row: entries of a row in the mean.  A launch of few rows is over when its longest row
// is: the row goes to as many groups as 2048 warps (the device's fill) leave room for; with one lane a group four pay at any size, eight up to 5000
// rows.  us per layer of 24, 4096 rows of 8 to 56 entries (of 32 in brackets), one group / this: 4 inputs 6.9 / 2.8 (4.5 / 2.8), 8 inputs 7.8 / 3.0
// (5.1 / 3.1), 16 inputs 5.3 / 3.4 (3.7 / 3.4), 32 inputs 5.2 / 4.2 (3.9 / 3.4), 64 inputs 7.1 / 5.8 (5.4 / 4.4); 700 rows, 128 inputs 6.3 / 4.5
// (4.9 / 3.4), 8 inputs 7.3 / 2.5.  More rows than that: 128 inputs, 4096 rows 8.5 with one group, 9.0 with two; two chunks, 2000 rows 4.8 and 5.0; 16 inputs,
// 16000 rows lanes of four inputs 8.2, two groups 8.4; 32 inputs, 10000 rows 7.2 with lanes of four inputs, 8.0 of eight, from 12000 on the other way round.
// A short row has nothing to share (one group / several: 3000 rows of 8, 16 inputs 3.3 / 3.9; 30000 of 8, 8 inputs 4.4 / 5.9; 2000 of 16, 32 inputs 3.5 / 3.9),
// and less of it where a lane holds few inputs or many groups wait already (8 inputs or 64: rows of 12 gain 4 to 20 %) and several chunks fill the device
// (1300 rows of 24, 384 inputs 4.0 / 4.8).
struct CsrGroups { int groups; bool narrow; };
inline CsrGroups csr_groups(int n, double per_row, int width, int chunks) {
    const bool between = width == 16 || width == 32;
    int groups = width <= 8 ? (n <= 5120 ? 8 : 4) : (int)std::min<int64_t>(8, 2048 * 32 / std::max<int64_t>(1, (int64_t)n * (width / 8)));
    if (width > 4 && per_row < (between ? 20 : width == 8 && n > 16384 ? 28 : 10)) groups = 1;
    if ((chunks == 2 && n > 1700) || (chunks > 1 && n > (chunks == 2 ? 1000 : 800) && per_row < 28)) groups = 1;
    return CsrGroups{groups, n <= (per_row < 20 ? 9200 : 11000)};
}
// ... entries of a row of layer l, as far as the offsets of the layers tell (which may lie in any order, and do not tell where the last one ends)
inline double csr_row(const int64_t* offset, int layers, int l, int n) {
    const int k = l + 1 < layers ? l : l - 1;
    const double entries = k < 0 ? 0.0 : (double)offset[k + 1] - (double)offset[k];
    return entries > 0 ? entries / n : 32.0;
}

// Units of a layer that does not fill the device, one per warp (see forward_split_kernel): first row * 8 + log2 of the groups of
// lanes that share a row.  off: offsets of the slices of 16 rows; a step is 8 entries of a row; `rows`: rows a warp works on at once with
// a group each; `slots`: warps that fit the device.  A slice's rows are split into as many parts as bring its steps down to the fewest
// that all units together leave room for.  Empty: nothing to gain by it.  So it is where the gathers of a launch outlast the round trips of its longest row (0.77 us each; 0.9 backward, where
// the update of the other copy goes over the same path): 30000 neurons, 6 inputs, 4 steps forward 6.82 us as it is, 7.00 split, 16384: 4.77 and
// 4.43; 16384, 28 inputs, backward 8.89 and 9.42, 10000: 8.03 and 7.01.
inline std::vector<unsigned> split_units(const std::vector<int>& off, int n, int rows, int row_bytes, int sms, int64_t slots, bool backward) {
    const int slices = (n + 15) / 16;
    int longest = 0;
    auto steps = [&](int s) { return (off[s + 1] - off[s]) / 128; };
    for (int s = 0; s < slices; ++s) longest = std::max(longest, steps(s));
    auto log_parts = [&](int s, int most) {
        int ls = rows > 16 ? 1 : 0;
        while ((rows >> (ls + 1)) >= 1 && ((steps(s) + (1 << ls) - 1) >> ls) > most) ++ls;
        return ls;
    };
    auto units_of = [&](int s, int ls) { return (std::min(16, n - s * 16) + (rows >> ls) - 1) / (rows >> ls); };
    if (longest * (backward ? 0.9 : 0.77) < (backward ? 2.0 : 1.0) * off[slices] / gathers_per_us(row_bytes, sms)) return {};
    int pick = longest;
    for (int most = longest - 1; most >= 1; --most) {
        int64_t units = 0;
        bool reached = true;
        for (int s = 0; s < slices && reached; ++s) {
            const int ls = log_parts(s, most);
            reached = ((steps(s) + (1 << ls) - 1) >> ls) <= most;
            units += units_of(s, ls);
        }
        if (!reached || units > slots) break;
        pick = most;
    }
    std::vector<unsigned> list;
    if (pick == longest) return list;
    for (int s = 0; s < slices; ++s) {
        const int ls = log_parts(s, pick);
        for (int u = 0; u < units_of(s, ls); ++u) list.push_back((unsigned)(s * 16 + u * (rows >> ls)) << 3 | (unsigned)ls);
    }
    return list;
}

// Whether the launches of layers that do not fill the device ask for the next launch's entries while they work (see forward_split_kernel).
// bytes: what a pass over the net walks: of an inference call the row-major copies, of a train step both copies, the activations and the
// deltas; width: columns of a train step's tiles, 0: inference.  A pass whose entries are near at hand pays for asking; how near they have to
// be was measured (us with / without, 24 to 480 layers of 640 to 6007 neurons, L2 126 MB): inference of 8 to 60 inputs 1.02 .. 1.07 up to 18 MB, 0.92 ..
// 0.99 from 23 MB on; train steps of 37 and 100 inputs 1.00 .. 1.01 up to 34 MB, 0.95 .. 1.00 from 47 MB (700 neurons x 100, 100 inputs,
// 99 MB: 0.88); of 8 to 28 inputs, whose launches wait for round trips and not for bytes, 1.00 .. 1.04 up to L2's size and 0.985 .. 1.02 beyond.
inline bool asks_ahead(int64_t bytes, int width, int64_t l2) { return width == 0 ? 6 * bytes > l2 : width >= 64 ? 3 * bytes > l2 : bytes > l2; }

}  // namespace sdnn_plan
