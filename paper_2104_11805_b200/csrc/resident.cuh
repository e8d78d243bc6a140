// Whole networks for many inputs in one launch: a CTA takes 4, 8, 12 or 16 inputs through all layers with their activations in its
// shared memory.
//
// Inference of nets whose layers fit (up to 8192 neurons).  The layer kernels gather every operand out of L2, which delivers 64 bytes
// per clock and SM, and run at that (66 operand bytes with what L1 happens to hold); shared memory delivers 128.  Inputs are independent, so a CTA needs nothing from another one: no tile, no
// launch and no barrier per layer on the device, and the network streams past out of L2, 6 bytes per entry and CTA.
//
// A slot holds one neuron's activations: P pieces of 4 inputs (16 bytes), each in a plane of its own.  A lane owns a row and reads P
// pieces per entry, so that the eight lanes that share a wavefront read eight slots: conflict-free where the slots differ modulo
// 8.  Random columns meet (2.5 wavefronts where one would do).  So the rows of a unit of 32 are chosen, and the order in which
// each reads its entries laid down, when the net is loaded: resident_order_kernel picks groups of eight rows whose columns
// spread evenly over the eight classes, resident_fill_kernel orders their entries step by step (resident.h).  1.06 wavefronts per
// eight entries are left at 32 random columns a row.  The order of a row's sum is all that this changes; it is the same for every
// width, so results do not depend on how a batch is cut into CTAs.  The layer launches keep the ascending order (in this one their gathers
// find less in L1: 4096 neurons, 128 inputs 4.91 -> 5.25 us a layer).  A row that has nothing to read in a step reads one of eight slots of zeros.
//
// Neurons are numbered by the place that their row was given: outputs are stored side by side, and columns name slots.
// Memory: a ring of slots.  A layer's outputs go behind its inputs; where both do not fit (4096 neurons, 8 inputs: 128 KB of
// inputs and 97 KB free) the last units' outputs wait in registers until every warp has read the layer.
// What bounds it is the shared-memory pipe (4096 neurons, 8 inputs a CTA: 0.27 wavefronts per entry and 8 inputs for operands, 0.05 for the
// entry itself; the pipe 86 % busy under ncu).  4096 x 120, 10000 inputs: 32.5 -> 25.6 ms,
// with dead inputs dropped, 5000 inputs a third of which survive: 9.58 -> 5.71; 2048 x 24, 2368 inputs: 34.9 -> 22.3 us a layer.
// 16 warps: with 20, 24 and 32 the same layer of 4096 takes 12, 10 and 6 % longer at 8 inputs a CTA (registers: fewer reads
// together), 4 inputs gain 4 % with 32.
#pragma once
#include "kernels.cuh"
#include "resident.h"

namespace sdnn_kernels {

using namespace sdnn_plan;
constexpr int RES_THREADS = RES_WARPS * 32;

// The entries: chunks of 4 per row, side by side for the 32 rows of a unit; unit u of layer k has chunks unit_at[k * units + u] ..
struct Resident {
    unsigned short* col;            // slot of each entry's column
    float* val;
    float* bias;                    // [layers][units * 32]
    int* unit_at;                   // [layers * units + 1]
    unsigned short* slot_of;        // [layers][n] slot of each neuron of the layer's output
    int* row_at;                    // [layers][units * 32] stored row (of the sliced copy) at each slot, -1: none
    int n, units;
};

struct ResidentArgs {
    Resident net;
    int from, to;                   // layers [from, to)
    int slots, cap;                 // of a layer; of the ring
    const float* x;                 // [inputs][n] activations before layer `from`, in neuron order
    float* y;                       // [inputs][n] ... after layer `to - 1`, or NULL
    int inputs, sms, width;         // see resident_share
    const int* list;                // inputs to take, *count of them (NULL: all)
    const int* count;
    int* nz_count;                  // [inputs] nonzero outputs, or NULL
    int* left;                      // inputs that are alive after layer `to - 1`, *n_left of them, or NULL
    int* n_left;
    int* live_hist;                 // dropping dead inputs: [layers] live inputs >= live_first after each layer, added up; else NULL
    int live_first;
    float clamp;
    int act;
};

__device__ __forceinline__ float4 res_ld(unsigned at) {
    float4 v;
    asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(at));
    return v;
}
__device__ __forceinline__ void res_st(unsigned at, const float4& v) {
    asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};" :: "r"(at), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w) : "memory");
}
// the network is read by every CTA at about the same time: L2 keeps it, L1 would not
__device__ __forceinline__ uint2 res_ld_col(const uint2* p) {
    uint2 v;
    asm volatile("ld.global.nc.L1::no_allocate.v2.u32 {%0, %1}, [%2];" : "=r"(v.x), "=r"(v.y) : "l"(p));
    return v;
}
__device__ __forceinline__ float4 res_ld_val(const float4* p) {
    float4 v;
    asm volatile("ld.global.nc.L1::no_allocate.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "l"(p));
    return v;
}

// HELD: units a warp keeps in registers (0: a layer's inputs and outputs both fit, and no slot number wraps).
template <int P, int HELD>
__global__ void __launch_bounds__(RES_THREADS, 1)
resident_infer_kernel(ResidentArgs a) {
    extern __shared__ __align__(128) unsigned char res_smem[];
    __shared__ int s_input[4 * P], s_count[4 * P];
    __shared__ unsigned s_live[3];
    constexpr int STRIDE = RES_WARPS;
    constexpr int AHEAD = P == 1 ? 4 : 2;                                    // chunks of entries on their way to a warp
    constexpr int TOGETHER = P > 2 ? 2 : 4;                                  // entries whose operands are read together
    int first, end;
    resident_share(a.count ? *a.count : a.inputs, a.sms, a.width, P, &first, &end);
    first += blockIdx.x * (4 * P);
    if (first >= end) return;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int n = a.net.n, units = a.net.units, rounds = (units + STRIDE - 1) / STRIDE;
    const unsigned base = (unsigned)__cvta_generic_to_shared(res_smem), ring = (unsigned)a.cap * 16u, layer = (unsigned)a.slots * 16u;
    auto wrap = [&](unsigned at) { return HELD ? min(at, at - ring) : at; };      // at < 2 * ring: the smaller one, as at - ring wraps below the ring's end

    if (threadIdx.x < 4 * P) {
        const int i = first + threadIdx.x;
        s_input[threadIdx.x] = i < end ? (a.list ? a.list[i] : i) : -1;
        s_count[threadIdx.x] = 0;
    }
    if (threadIdx.x < 3) s_live[threadIdx.x] = 0u;
    __syncthreads();

    // inputs
    unsigned in = 0;
    {
        const unsigned short* map = a.from ? a.net.slot_of + (size_t)(a.from - 1) * n : nullptr;
        for (int j = threadIdx.x; j < n; j += RES_THREADS) {
            const unsigned at = base + (map ? map[j] : j) * 16u;
#pragma unroll
            for (int p = 0; p < P; ++p) {
                float v[4];
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const int b = s_input[4 * p + i];
                    v[i] = b >= 0 ? __ldcs(a.x + (size_t)b * n + j) : 0.0f;
                }
                res_st(at + p * ring, make_float4(v[0], v[1], v[2], v[3]));
            }
        }
        for (int j = n + threadIdx.x; j < a.slots; j += RES_THREADS)
#pragma unroll
            for (int p = 0; p < P; ++p) res_st(base + j * 16u + p * ring, make_float4(0.f, 0.f, 0.f, 0.f));
    }

    // The entries reach a warp AHEAD chunks before it works on them: `q` is the chunk to fetch next, of the unit that ends at `q_end`; (r, r_end) those
    // of the unit after it.
    const uint2* col = reinterpret_cast<const uint2*>(a.net.col) + lane;
    const float4* val = reinterpret_cast<const float4*>(a.net.val) + lane;
    const int last_unit = a.to * units - 1;
    int f_unit = a.from * units + warp, f_round = 0;
    const bool works = warp < units;
    int q = 0, q_end = 0, r = 0, r_end = 0;
    auto after = [&]() {                                                     // the unit after f_unit in this warp's walk
        ++f_round;
        f_unit += STRIDE;
        if (f_round * STRIDE + warp >= units) { f_unit += units - f_round * STRIDE; f_round = 0; }
        const int u = min(f_unit, last_unit);
        r = a.net.unit_at[u]; r_end = a.net.unit_at[u + 1];
    };
    uint2 ec[AHEAD];
    float4 ew[AHEAD];
    auto fetch = [&](uint2& c, float4& w) {
        c = res_ld_col(col + (size_t)q * 32); w = res_ld_val(val + (size_t)q * 32);
        if (++q == q_end) { q = r; q_end = r_end; after(); }
    };
    int chunks = 0, next_chunks = 0;
    float bias = 0.0f, next_bias = 0.0f;
    auto look = [&](int unit) {                                              // shape and bias of a unit that is worked on later
        const int u = min(unit, last_unit);
        next_chunks = a.net.unit_at[u + 1] - a.net.unit_at[u];
        next_bias = a.net.bias[(size_t)u * 32 + lane];
    };
    if (works) {
        q = a.net.unit_at[f_unit]; q_end = a.net.unit_at[f_unit + 1];
        look(f_unit);
        after();
#pragma unroll
        for (int i = 0; i < AHEAD; ++i) fetch(ec[i], ew[i]);
    }
    __syncthreads();

    const bool track = a.live_hist != nullptr;
    unsigned valid = 0u, counted = 0u, live = 0u;      // bit b: input b of this CTA exists; belongs to the last tile; is alive
#pragma unroll
    for (int b = 0; b < 4 * P; ++b) {
        valid |= (s_input[b] >= 0 ? 1u : 0u) << b;
        counted |= (s_input[b] >= a.live_first ? 1u : 0u) << b;
    }
    live = valid;

    for (int k = a.from; k < a.to; ++k) {
        const unsigned out = in + layer < ring ? in + layer : in + layer - ring;
        const unsigned from = base + in;
        unsigned mine = 0u;                                                  // bits of inputs that a row of this thread keeps alive
        // one unit: 32 rows, a lane each
        auto work = [&](int u, float4 (&acc)[P]) {
            chunks = next_chunks; bias = next_bias;
            look(k * units + (u + STRIDE < units ? u + STRIDE : units + warp));
#pragma unroll
            for (int p = 0; p < P; ++p) acc[p] = make_float4(bias, bias, bias, bias);
            auto chunk = [&](uint2& c, float4& w) {
                const float4 wv = w;
                unsigned at[4] = {(c.x & 0xffffu) * 16u, (c.x >> 16) * 16u, (c.y & 0xffffu) * 16u, (c.y >> 16) * 16u};
#pragma unroll
                for (int e = 0; e < 4; ++e) at[e] = HELD ? base + wrap(at[e] + in) : at[e] + from;
                fetch(c, w);
                const float we[4] = {wv.x, wv.y, wv.z, wv.w};
#pragma unroll
                for (int e = 0; e < 4; e += TOGETHER) {
                    float4 x[TOGETHER][P];
#pragma unroll
                    for (int i = 0; i < TOGETHER; ++i)
#pragma unroll
                        for (int p = 0; p < P; ++p) x[i][p] = res_ld(at[e + i] + p * ring);
#pragma unroll
                    for (int i = 0; i < TOGETHER; ++i)
#pragma unroll
                        for (int p = 0; p < P; ++p) f4_fma(we[e + i], x[i][p], acc[p]);
                }
            };
            int t = chunks;
            for (; t >= AHEAD; t -= AHEAD)
#pragma unroll
                for (int i = 0; i < AHEAD; ++i) chunk(ec[i], ew[i]);
            for (; t; --t) {                                                 // the chunks that are on their way move up
                chunk(ec[0], ew[0]);
                const uint2 c = ec[0];
                const float4 w = ew[0];
#pragma unroll
                for (int i = 0; i + 1 < AHEAD; ++i) { ec[i] = ec[i + 1]; ew[i] = ew[i + 1]; }
                ec[AHEAD - 1] = c; ew[AHEAD - 1] = w;
            }
            const bool row = u * RES_UNIT + lane < n;
#pragma unroll
            for (int p = 0; p < P; ++p) {
                f4_activate(acc[p], a.act, a.clamp);
                if (!row) acc[p] = make_float4(0.f, 0.f, 0.f, 0.f);
                mine |= f4_nonzero_bits(acc[p]) << (4 * p);
            }
        };
        auto store = [&](int u, const float4 (&acc)[P]) {
            const unsigned at = base + wrap(out + (unsigned)(u * RES_UNIT + lane) * 16u);
#pragma unroll
            for (int p = 0; p < P; ++p) res_st(at + p * ring, acc[p]);
        };
        auto zeros = [&]() {
            if (warp == RES_WARPS - 1 && lane < RES_CLASSES)
#pragma unroll
                for (int p = 0; p < P; ++p) res_st(base + wrap(out + (unsigned)(units * RES_UNIT + lane) * 16u) + p * ring, make_float4(0.f, 0.f, 0.f, 0.f));
        };
        for (int i = 0; i < rounds - HELD; ++i) {
            const int u = i * STRIDE + warp;
            if (u >= units) break;
            float4 acc[P];
            work(u, acc);
            store(u, acc);
        }
        float4 held[HELD ? HELD : 1][P];
#pragma unroll
        for (int i = 0; i < HELD; ++i) {
            const int u = (rounds - HELD + i) * STRIDE + warp;
            if (u < units) work(u, held[i]);
        }
        if (!HELD) zeros();
        if (track) {
            mine = __reduce_or_sync(0xffffffffu, mine);
            if (lane == 0 && mine) atomicOr(&s_live[k % 3], mine);
            if (threadIdx.x == 0) s_live[(k + 1) % 3] = 0u;                  // last read before the barrier of layer k - 1
        }
        __syncthreads();
        if (HELD) {
#pragma unroll
            for (int i = 0; i < HELD; ++i) {
                const int u = (rounds - HELD + i) * STRIDE + warp;
                if (u < units) store(u, held[i]);
            }
            zeros();
            __syncthreads();
        }
        in = out;
        if (track) {
            live = s_live[k % 3] & valid;
            if (threadIdx.x == 0 && (live & counted)) atomicAdd(&a.live_hist[k], __popc(live & counted));
            if (!live) break;                                                // zeros from here on: what this layer left are the outputs
        }
    }

    if (a.left && threadIdx.x < 4 * P && (live >> threadIdx.x & 1u)) a.left[atomicAdd(a.n_left, 1)] = s_input[threadIdx.x];
    if (!a.y && !a.nz_count) return;
    const unsigned short* map = a.net.slot_of + (size_t)(a.to - 1) * n;
    int some[4 * P];
#pragma unroll
    for (int b = 0; b < 4 * P; ++b) some[b] = 0;
    for (int j = threadIdx.x; j < n; j += RES_THREADS) {
        const unsigned at = base + wrap(in + map[j] * 16u);
#pragma unroll
        for (int p = 0; p < P; ++p) {
            const float4 x = res_ld(at + p * ring);
            const float v[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int b = s_input[4 * p + i];
                if (a.y && b >= 0) __stcs(a.y + (size_t)b * n + j, v[i]);
                some[4 * p + i] += v[i] != 0.0f ? 1 : 0;
            }
        }
    }
    if (!a.nz_count) return;
#pragma unroll
    for (int b = 0; b < 4 * P; ++b) {
        const int s = __reduce_add_sync(0xffffffffu, some[b]);
        if (lane == 0 && s) atomicAdd(&s_count[b], s);
    }
    __syncthreads();
    if (threadIdx.x < 4 * P && s_input[threadIdx.x] >= 0) a.nz_count[s_input[threadIdx.x]] = s_count[threadIdx.x];
}

// ---------------------------------------------------------------------------------------------
// Ids of the nonzero outputs of `cnt` inputs, from the outputs themselves: a block per input, 32 neurons a warp at a time; offs as
// nz_scan_inputs_kernel left them.
__global__ void __launch_bounds__(256)
nz_fill_rows_kernel(const float* __restrict__ y, const long long* __restrict__ offs, int* __restrict__ out, long long capacity, int n) {
    __shared__ int part[2][8];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, b = blockIdx.x;
    const float* row = y + (size_t)b * n;
    long long pos = offs[b];
    for (int i0 = 0, turn = 0; i0 < n; i0 += 1024, turn ^= 1) {      // four ids a thread
        const int i = i0 + threadIdx.x * 4;
        unsigned m = 0u;
#pragma unroll
        for (int e = 0; e < 4; ++e) if (i + e < n && row[i + e] != 0.0f) m |= 1u << e;
        int before = __popc(m);
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int v = __shfl_up_sync(0xffffffffu, before, o);
            if (lane >= o) before += v;
        }
        if (lane == 31) part[turn][warp] = before;
        __syncthreads();
        int skip = 0, all = 0;
#pragma unroll
        for (int q = 0; q < 8; ++q) { if (q < warp) skip += part[turn][q]; all += part[turn][q]; }
        long long at = pos + skip + before - __popc(m);
        while (m) {
            if (at < capacity) out[at] = i + __ffs(m) - 1;
            ++at;
            m &= m - 1;
        }
        pos += all;
    }
}

// ---------------------------------------------------------------------------------------------
// Set-up, all layers at once.  place0 (or NULL: identity) is where a neuron's row stands before rows are grouped; grouping moves it
// among the RES_BLOCK rows around it, to a place of the same class: columns have their classes before any layer is grouped.
struct ResidentSetup {
    const Sliced* rows;                 // [layers] sliced copies
    const float* const* bias;           // [layers] in stored order
    const unsigned short* row0;         // [layers][n] stored row at each place, or NULL: identity
    const unsigned short* place0;       // [layers][n] place of each neuron, or NULL: identity
    unsigned char* const* order;        // [layers] which of a row's entries (by their places in the sliced copy) is read at each place
    int layer0;                         // first layer of the launch
};

// A block of RES_BLOCK rows, a group of eight after the other: rows of two groups change places while that spreads the groups' columns
// more evenly over the eight classes (fourth powers of the distances from the mean: the largest one decides how many steps of a group take
// two wavefronts).  Every group meets every other one RES_PASSES times, a row only rows of its own length in chunks and of its own class of
// place.  32 random columns a row: 1.25 wavefronts per step as the rows come, 1.069, 1.060, 1.057 after one, two, three passes;
// 1.087 among 256 rows.  Rows beyond the last whole group keep their places.
constexpr int RES_PASSES = 3;
__global__ void __launch_bounds__(RES_BLOCK)
resident_order_kernel(Resident net, ResidentSetup s) {
    constexpr int GROUPS = RES_BLOCK / 8;
    __shared__ uint2 s_cnt[RES_BLOCK];                          // columns of each row in each class, a byte each
    __shared__ unsigned char s_chunks[RES_BLOCK];
    __shared__ unsigned short s_pick[RES_BLOCK];                // row at each place
    __shared__ short s_sum[GROUPS][8];                          // columns of each group in each class
    const int k = s.layer0 + blockIdx.y, n = net.n, p0 = blockIdx.x * RES_BLOCK, p = p0 + threadIdx.x;
    const Sliced m = s.rows[k];
    const unsigned short* classes = k && s.place0 ? s.place0 + (size_t)(k - 1) * n : nullptr;
    int len = 0;
    unsigned lo = 0u, hi = 0u;
    if (p < n) {
        const int row = s.row0 ? s.row0[(size_t)k * n + p] : p;
        len = m.len[row];
        const int at = m.slice_off[row / SLICE] + (row % SLICE) * 4;
        for (int q = 0; q < len; ++q) {
            const int col = load_idx1(m, at + (q >> 2) * CHUNK_ROW + (q & 3)), c = (classes ? classes[col] : col) & 7;
            if (c < 4) lo += 1u << (8 * c); else hi += 1u << (8 * (c - 4));
        }
    }
    s_cnt[threadIdx.x] = make_uint2(lo, hi);
    s_chunks[threadIdx.x] = (unsigned char)((len + 3) / 4);
    s_pick[threadIdx.x] = (unsigned short)threadIdx.x;
    __syncthreads();
    auto count = [](const uint2& v, int c) { return (int)((c < 4 ? v.x >> (8 * c) : v.y >> (8 * (c - 4))) & 0xffu); };
    const int g_own = threadIdx.x >> 3, l = threadIdx.x & 7;
    {
        int v = 0;
        for (int r = 0; r < 8; ++r) v += count(s_cnt[g_own * 8 + r], l);
        s_sum[g_own][l] = (short)v;
    }
    __syncthreads();
    const int whole = min(RES_BLOCK, n - p0) / 8;               // groups of this block
    for (int pass = 0; pass < RES_PASSES; ++pass)
        for (int d = 1; d < GROUPS; ++d) {
            // groups g and g ^ d, eight threads a pair, one for each place
            const int bit = 31 - __clz(d), pair = g_own, g = ((pair >> bit) << (bit + 1)) | (pair & ((1 << bit) - 1)), h = g ^ d;
            if (pair < GROUPS / 2 && h < whole) {
                const unsigned lanes = 0xffu << (threadIdx.x & 24);
                const int a = s_pick[g * 8 + l], b = s_pick[h * 8 + l];
                const uint2 ca = s_cnt[a], cb = s_cnt[b];
                float before = 0.0f, after = 0.0f;
                int sg = 0, sh = 0, dd = 0;
#pragma unroll
                for (int c = 0; c < 8; ++c) { sg += s_sum[g][c]; sh += s_sum[h][c]; dd += count(ca, c) - count(cb, c); }
                const float mg = sg * 0.125f, mh = sh * 0.125f, ng = (sg - dd) * 0.125f, nh = (sh + dd) * 0.125f;
#pragma unroll
                for (int c = 0; c < 8; ++c) {
                    const int e = count(ca, c) - count(cb, c), x = s_sum[g][c], y = s_sum[h][c];
                    float v = (x - mg) * (x - mg), w = (y - mh) * (y - mh);
                    before += v * v + w * w;
                    v = (x - e - ng) * (x - e - ng); w = (y + e - nh) * (y + e - nh);
                    after += v * v + w * w;
                }
                if (s_chunks[a] != s_chunks[b]) after = 3e38f;
                const unsigned gain = after < before ? (__float_as_uint(after) & ~7u) | (unsigned)l : 0xffffffffu;      // after >= 0
                unsigned best = gain;
#pragma unroll
                for (int o = 1; o < 8; o <<= 1) best = min(best, __shfl_xor_sync(lanes, best, o));
                if (best != 0xffffffffu && best == gain) {      // one thread: the place is part of the number
                    s_pick[g * 8 + l] = (unsigned short)b; s_pick[h * 8 + l] = (unsigned short)a;
#pragma unroll
                    for (int c = 0; c < 8; ++c) {
                        const int e = count(ca, c) - count(cb, c);
                        s_sum[g][c] -= (short)e; s_sum[h][c] += (short)e;
                    }
                }
            }
            __syncthreads();
        }
    if (p < net.units * RES_UNIT) {
        int at_row = -1;
        if (p < n) {
            const int from = p0 + s_pick[threadIdx.x];
            at_row = s.row0 ? s.row0[(size_t)k * n + from] : from;
            net.slot_of[(size_t)k * n + (m.out ? m.out[at_row] : at_row)] = (unsigned short)p;
        }
        net.row_at[(size_t)k * net.units * RES_UNIT + p] = at_row;
    }
}

// A unit per block of one warp: the order in which its rows read their entries.  list: entries of each row, class by class.
__global__ void __launch_bounds__(32)
resident_fill_kernel(Resident net, ResidentSetup s, int pitch) {
    extern __shared__ unsigned char res_list[];                 // [32][pitch] positions of a row's entries, at most RES_MAX_ROW
    const int k = s.layer0 + blockIdx.y, u = blockIdx.x, lane = threadIdx.x, n = net.n, grp = lane >> 3;
    const Sliced m = s.rows[k];
    const unsigned short* slots = k ? net.slot_of + (size_t)(k - 1) * n : nullptr;
    const int place = u * RES_UNIT + lane;
    const int row = net.row_at[(size_t)k * net.units * RES_UNIT + place];
    net.bias[(size_t)k * net.units * RES_UNIT + place] = row >= 0 ? s.bias[k][row] : 0.0f;
    const int len = row >= 0 ? m.len[row] : 0, at = row >= 0 ? m.slice_off[row / SLICE] + (row % SLICE) * 4 : 0;
    unsigned char* list = res_list + lane * pitch;
    auto entry = [&](int q) { return at + (q >> 2) * CHUNK_ROW + (q & 3); };
    auto slot = [&](int q) { const int c = load_idx1(m, entry(q)); return slots ? (int)slots[c] : c; };
    unsigned long long left = 0, next = 0;                      // byte c: entries of class c not read yet; place of the next one in the list
    for (int q = 0; q < len; ++q) left += 1ull << (8 * (slot(q) & 7));
    {
        unsigned long long run = 0;
        for (int c = 0; c < 8; ++c) { next |= run << (8 * c); run += (left >> (8 * c)) & 0xffu; }
        unsigned long long put = next;
        for (int q = 0; q < len; ++q) {
            const int c = slot(q) & 7;
            list[(put >> (8 * c)) & 0xffu] = (unsigned char)q;
            put += 1ull << (8 * c);
        }
    }
    int total[8];
#pragma unroll
    for (int c = 0; c < 8; ++c) {
        int v = (int)((left >> (8 * c)) & 0xffu);
        v += __shfl_xor_sync(0xffffffffu, v, 1); v += __shfl_xor_sync(0xffffffffu, v, 2); v += __shfl_xor_sync(0xffffffffu, v, 4);
        total[c] = v;
    }
    const int q0 = net.unit_at[k * net.units + u], steps = 4 * (net.unit_at[k * net.units + u + 1] - q0);
    int togo = len;
    for (int t = 0; t < steps; ++t) {
        unsigned long long have = 0;
#pragma unroll
        for (int c = 0; c < 8; ++c)
            have |= (unsigned long long)((__ballot_sync(0xffffffffu, ((left >> (8 * c)) & 0xffu) != 0) >> (8 * grp)) & 0xffu) << (8 * c);
        const unsigned must = (__ballot_sync(0xffffffffu, togo > 0 && togo >= steps - t) >> (8 * grp)) & 0xffu;
        const unsigned of_row = resident_step(have, total, must, steps - t);
        const int c = (int)((of_row >> (4 * (lane & 7))) & 15u);
        int to_slot = net.units * RES_UNIT;
        float w = 0.0f;
        if (c != 15) {
            const int q = list[(next >> (8 * c)) & 0xffu];
            next += 1ull << (8 * c);
            left -= 1ull << (8 * c);
            s.order[k][entry(len - togo)] = (unsigned char)q;
            --togo;
            to_slot = slot(q);
            w = m.val[entry(q)];
        } else to_slot += resident_idle_class(of_row, lane & 7);
#pragma unroll
        for (int d = 0; d < 8; ++d)
#pragma unroll
            for (int r = 0; r < 8; ++r) total[d] -= ((of_row >> (4 * r)) & 15u) == (unsigned)d ? 1 : 0;
        const size_t o = ((size_t)(q0 + (t >> 2)) * 32 + lane) * 4 + (t & 3);
        net.col[o] = (unsigned short)to_slot;
        net.val[o] = w;
        __syncwarp();
    }
}

// The sliced copies once more with their rows' entries in that order (a warp a row), for handles that drop dead inputs: where a batch is
// too small to be dropped this way but goes this way without dropping, the layer launches read these, so that dropping changes no bit.
__global__ void __launch_bounds__(256)
resident_reorder_kernel(ResidentSetup s, int n, int* const* idx, float* const* val) {
    const int k = s.layer0 + blockIdx.y, row = blockIdx.x * 8 + (threadIdx.x >> 5);
    if (row >= n) return;
    const Sliced m = s.rows[k];
    const int len = m.len[row], at = m.slice_off[row / SLICE] + (row % SLICE) * 4;
    auto entry = [&](int q) { return at + (q >> 2) * CHUNK_ROW + (q & 3); };
    for (int q = threadIdx.x & 31; q < len; q += 32) {
        const int from = entry(s.order[k][entry(q)]);
        if (m.idx16) reinterpret_cast<unsigned short*>(idx[k])[entry(q)] = (unsigned short)load_idx1(m, from);
        else idx[k][entry(q)] = load_idx1(m, from);
        val[k][entry(q)] = m.val[from];
    }
}

// New values and biases, from the sliced copy: a unit per block of one warp.
__global__ void __launch_bounds__(32)
resident_refill_kernel(Resident net, ResidentSetup s) {
    const int k = s.layer0, u = blockIdx.x, lane = threadIdx.x, place = u * RES_UNIT + lane;
    const Sliced m = s.rows[k];
    const int row = net.row_at[(size_t)k * net.units * RES_UNIT + place];
    net.bias[(size_t)k * net.units * RES_UNIT + place] = row >= 0 ? s.bias[k][row] : 0.0f;
    if (row < 0) return;
    const int at = m.slice_off[row / SLICE] + (row % SLICE) * 4;
    const int q0 = net.unit_at[k * net.units + u], steps = 4 * (net.unit_at[k * net.units + u + 1] - q0);
    for (int t = 0, q = 0; t < steps; ++t) {
        const size_t o = ((size_t)(q0 + (t >> 2)) * 32 + lane) * 4 + (t & 3);
        if (net.col[o] >= net.units * RES_UNIT) continue;      // a step in which the row waits
        const int from = s.order[k][at + (q >> 2) * CHUNK_ROW + (q & 3)];
        net.val[o] = m.val[at + (from >> 2) * CHUNK_ROW + (from & 3)];
        ++q;
    }
}

}  // namespace sdnn_kernels
