// Rules of the launches that need no device: plain host code, so that they can be looked at without one.
#pragma once
#include <stdint.h>

#include <algorithm>

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
inline TileShape tile_shape(int cnt, int64_t elems, bool windows) {
    TileShape best{std::min(padded_width(cnt), 256), padded_width(cnt)};
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
struct GraphKey { int cw = 0, cols = 0, used = 0, pdl = 0; bool track = false; };
inline int pick_graph(const GraphKey* have, const int64_t* asked, int n, GraphKey& want, bool& make) {      // asked[q] = 0: empty
    int room = -1, serves = -1, oldest = 0;
    make = false;
    for (int q = 0; q < n; ++q) {
        if (!asked[q]) { if (room < 0) room = q; continue; }
        const GraphKey& g = have[q];
        if (g.cw == want.cw && g.cols == want.cols && g.pdl == want.pdl && g.track == want.track && g.used >= want.used) {
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

}  // namespace sdnn_plan
