// Device kernels of the sparse-DNN SGD hot path (sm_100a).
//
// Tiles.  Activations x^k, deltas and the partial products S = W^T delta live in neuron-major tiles
// X[i*ld + b] (neuron i, input b; ld = padded batch), so that the row of X gathered for one stored entry
// W(i,j) is contiguous.  A lane holds V = 8 batch entries of a row (one 256-bit access; V = 4 only for tiles
// of 4 columns), a row is shared by G = ld / V lanes, and a warp works on 32/G matrix rows at once.  Tiles
// wider than 256 inputs are processed in chunks of 256 (blockIdx.y).
//
// Stored entries.  These kernels are bound by the memory requests an SM can make per stored entry, not by
// bytes: the gather of a tile row costs one request whatever its width up to 64 bytes (a store that leaves
// holes in a 32-byte sector costs several), and with
// plain CSR the index and value loads of the row groups of a warp would cost as much again, because each row
// sits in a different 128-byte line.  The entries are therefore kept in slices of 16 rows, interleaved in
// chunks of 4:
//     entry q of row i  ->  slice_off[i/16] + (q/4)*64 + (i%16)*4 + q%4          (element offset)
// so that the chunks (16 bytes of values, 8 or 16 bytes of indices: the index array holds 16-bit indices for nets of at
// most 65536 neurons, template parameter I16 of the layer kernels) the row groups of a warp read in one step are
// contiguous.  A slice is padded
// to the longest of its rows rounded up to 8; padding has index 0 and value 0 and is never updated.  The
// transposed matrix (columns as "rows", for the backward product without atomics) uses the same layout over
// the columns sorted by descending length.
//
// Equations (paper, Section 3.2): forward x^k = f(W^k x^{k-1} + b^k); recursion
// delta^{k-1} = (W^k)^T delta^k (.) f'(z^{k-1}); update W^k(j,i) -= eta delta^k(j) x^{k-1}(i)
// on stored entries.  Only x^k is stored: with f = clamp to [0,c], f'(z) = [0 < x < c].
#pragma once
#include <cuda.h>
#include <cuda_runtime.h>
#include <stdint.h>

namespace sdnn_kernels {

struct StepParams {     // written by start_step_kernel at the start of each train step; read by the graph's kernels
    float eta;          // learning rate
    float inv_b;        // 1 / B
    int   batch;        // B (valid inputs; the tile is zero-padded to ld)
    int   pad;
};

constexpr int SLICE = 16;            // rows per slice
constexpr int CHUNK_ROW = SLICE * 4; // elements of one chunk over the rows of a slice

// One matrix in sliced layout.  `order` is NULL for the row-major copy (unit u is row u); for the
// transposed copy it lists the matrix column each unit stands for.
struct Sliced {
    const int* slice_off;   // [ceil(n/16) + 1] element offsets of the slices, multiples of 128
    const int* len;         // [n] stored entries of each unit
    const int* idx;         // gathered tile row of each entry (column index; row index in the transposed copy);
                            // with idx16 set the array holds 16-bit unsigned indices instead (nets of at most 65536 neurons)
    float*     val;
    const int* order;
    int idx16;
    const int* out;         // tile row that stored row u stands for (NULL: row u): ragged layers, whose rows are stored by length,
                            // and layers stored group by group (neurons numbered by the next layer's grouping)
};

__device__ __forceinline__ float4 ld_f4(const float* p) { return *reinterpret_cast<const float4*>(p); }
__device__ __forceinline__ void st_f4(float* p, float4 v) { *reinterpret_cast<float4*>(p) = v; }

// read-only gather of a tile row segment (goes through the non-coherent path)
__device__ __forceinline__ float4 gather_f4(const float* p) { return __ldg(reinterpret_cast<const float4*>(p)); }

// 128-bit vector reduction into global memory (sm_90+): four fp32 adds in one L2 operation
__device__ __forceinline__ void red_add_f4(float* p, float4 v) {
    asm volatile("red.relaxed.gpu.global.add.v4.f32 [%0], {%1, %2, %3, %4};"
                 :: "l"(p), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w) : "memory");
}

// asks for `bytes` (a multiple of 16, address 16-byte aligned) to be brought into L2; no destination, no wait
__device__ __forceinline__ void prefetch_l2(const void* p, unsigned bytes) {
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" :: "l"(p), "r"(bytes) : "memory");
}

// programmatic dependent launch: wait for the kernels this one depends on / let the next one start its prologue.
// The layer kernels take `pdl`: 0 = launched without the attribute (no wait, no release); 1 = wait, release the next
// launch at the end; 2 = wait, release it right after the wait (its CTAs then move into SM slots as they fall free and
// do everything that does not depend on this launch - shapes, first indices - under this launch's tail).  Whatever a
// kernel reads before its wait must not be written by the launch before it: slice offsets, lengths, order, indices,
// (forward) the bias and (column units of the backward pass) the step parameters and the rows of x^{k-1}, which the
// forward pass of the same step wrote, qualify; values, the delta tiles and counters do not.
__device__ __forceinline__ void grid_dependency_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void grid_launch_dependents() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

__device__ __forceinline__ float clampf(float z, float c) { return fminf(fmaxf(z, 0.0f), c); }
__device__ __forceinline__ float dmask(float x, float c) { return (x > 0.0f && x < c) ? 1.0f : 0.0f; }

// Activations (cfg.activation): 0 = ReLU clamped at c, f'(z) = [0 < x < c]; 1 = sigmoid (the activation of the
// paper's experiments, Section 6), f'(z) = x (1 - x).  Both derivatives are functions of the stored output x.
constexpr int ACT_CLAMPED_RELU = 0, ACT_SIGMOID = 1;
__device__ __forceinline__ float activate(float z, int act, float c) {
    // sigmoid with the hardware's exp2 and reciprocal approximations (relative error about 1e-6 for |z| <= 20, against a
    // parity bar of 1e-4): the accurate expf and division cost a forward launch of 16 inputs 10 % of its time, all of it
    // in the tail of the launch where nothing else runs
    return act == ACT_SIGMOID ? __fdividef(1.0f, 1.0f + __expf(-z)) : clampf(z, c);
}
__device__ __forceinline__ float derivative(float x, int act, float c) {
    return act == ACT_SIGMOID ? x * (1.0f - x) : dmask(x, c);
}

// address of tile row `r` (r * pitch below 2^32): one 32 x 32 -> 64 bit multiply-add
__device__ __forceinline__ const float* tile_row(const float* base, int r, unsigned pitch_bytes) {
    unsigned long long out;
    asm("mad.wide.u32 %0, %1, %2, %3;" : "=l"(out) : "r"(r), "r"(pitch_bytes), "l"(base));
    return reinterpret_cast<const float*>(out);
}
__device__ __forceinline__ float* tile_row(float* base, int r, unsigned pitch_bytes) {
    unsigned long long out;
    asm("mad.wide.u32 %0, %1, %2, %3;" : "=l"(out) : "r"(r), "r"(pitch_bytes), "l"(base));
    return reinterpret_cast<float*>(out);
}

// ---------------------------------------------------------------------------------------------
// The V batch entries a lane holds of one tile row.
template <int V> struct Lane;
template <> struct Lane<4> { float4 a; };
template <> struct Lane<8> { float4 a, b; };

__device__ __forceinline__ void lane_fill(Lane<4>& v, float s) { v.a = make_float4(s, s, s, s); }
__device__ __forceinline__ void lane_fill(Lane<8>& v, float s) { v.a = make_float4(s, s, s, s); v.b = v.a; }

__device__ __forceinline__ void lane_load(Lane<4>& v, const float* p) { v.a = ld_f4(p); }
__device__ __forceinline__ void lane_load(Lane<8>& v, const float* p) {      // one 256-bit load (p 32-byte aligned)
    asm volatile("ld.global.v8.f32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                 : "=f"(v.a.x), "=f"(v.a.y), "=f"(v.a.z), "=f"(v.a.w), "=f"(v.b.x), "=f"(v.b.y), "=f"(v.b.z), "=f"(v.b.w) : "l"(p) : "memory");
}
__device__ __forceinline__ void lane_gather(Lane<4>& v, const float* p) { v.a = gather_f4(p); }
__device__ __forceinline__ void lane_gather(Lane<8>& v, const float* p) {    // read-only path, one 256-bit load
    asm volatile("ld.global.nc.v8.f32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                 : "=f"(v.a.x), "=f"(v.a.y), "=f"(v.a.z), "=f"(v.a.w), "=f"(v.b.x), "=f"(v.b.y), "=f"(v.b.z), "=f"(v.b.w) : "l"(p));
}
// The same gather past L1 (cached in L2 only).  For rows of up to 64 bytes out of a tile that no L1 can hold, a probe of
// nothing but such gathers runs 6 % faster this way (0.82 against 0.77 rows per clock and SM) and the forward launches of
// 16 inputs 2 %; wider rows, which several lanes read side by side, and the backward launches lose by it.
// (Only for layers without padding entries: those all point at tile row 0, which L1 absorbs and one L2 slice would not.)
template <bool PAST_L1> __device__ __forceinline__ void lane_gather_sel(Lane<4>& v, const float* p) { v.a = gather_f4(p); }
template <bool PAST_L1> __device__ __forceinline__ void lane_gather_sel(Lane<8>& v, const float* p) {
    if (PAST_L1)
        asm volatile("ld.global.cg.v8.f32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                     : "=f"(v.a.x), "=f"(v.a.y), "=f"(v.a.z), "=f"(v.a.w), "=f"(v.b.x), "=f"(v.b.y), "=f"(v.b.z), "=f"(v.b.w) : "l"(p));
    else lane_gather(v, p);
}
__device__ __forceinline__ void lane_store(float* p, const Lane<4>& v) { st_f4(p, v.a); }
__device__ __forceinline__ void lane_store(float* p, const Lane<8>& v) {
    asm volatile("st.global.v8.f32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};"
                 :: "l"(p), "f"(v.a.x), "f"(v.a.y), "f"(v.a.z), "f"(v.a.w), "f"(v.b.x), "f"(v.b.y), "f"(v.b.z), "f"(v.b.w) : "memory");
}

// acc += w * x with packed two-wide fp32 FMAs (sm_100): half the issue slots of scalar FMAs
__device__ __forceinline__ void f4_fma(float w, const float4& x, float4& a) {
    const float2 ww = make_float2(w, w);
    const float2 lo = __ffma2_rn(ww, make_float2(x.x, x.y), make_float2(a.x, a.y));
    const float2 hi = __ffma2_rn(ww, make_float2(x.z, x.w), make_float2(a.z, a.w));
    a = make_float4(lo.x, lo.y, hi.x, hi.y);
}
__device__ __forceinline__ void lane_fma(float w, const Lane<4>& x, Lane<4>& acc) { f4_fma(w, x.a, acc.a); }
__device__ __forceinline__ void lane_fma(float w, const Lane<8>& x, Lane<8>& acc) { f4_fma(w, x.a, acc.a); f4_fma(w, x.b, acc.b); }

// Partial dot product of one lane: its batch columns of delta (d) against those of x, even and odd columns in
// the two halves of packed FMAs, added at the end.  Written with explicit roundings and a fixed order so that the
// row pass and the column pass, which swap the roles of the gathered and the resident operand, produce the same
// bits (a*b and fma(a,b,c) are symmetric in a and b).
__device__ __forceinline__ float lane_dot(const Lane<4>& d, const Lane<4>& x) {
    float2 p = __fmul2_rn(make_float2(d.a.x, d.a.y), make_float2(x.a.x, x.a.y));
    p = __ffma2_rn(make_float2(d.a.z, d.a.w), make_float2(x.a.z, x.a.w), p);
    return __fadd_rn(p.x, p.y);
}
__device__ __forceinline__ float lane_dot(const Lane<8>& d, const Lane<8>& x) {
    float2 p = __fmul2_rn(make_float2(d.a.x, d.a.y), make_float2(x.a.x, x.a.y));
    p = __ffma2_rn(make_float2(d.a.z, d.a.w), make_float2(x.a.z, x.a.w), p);
    p = __ffma2_rn(make_float2(d.b.x, d.b.y), make_float2(x.b.x, x.b.y), p);
    p = __ffma2_rn(make_float2(d.b.z, d.b.w), make_float2(x.b.z, x.b.w), p);
    return __fadd_rn(p.x, p.y);
}

// d *= f'(z) with f' taken from the stored output x
__device__ __forceinline__ void f4_mask(float4& d, const float4& x, int act, float c) {
    d.x *= derivative(x.x, act, c); d.y *= derivative(x.y, act, c); d.z *= derivative(x.z, act, c); d.w *= derivative(x.w, act, c);
}
__device__ __forceinline__ void lane_mask(Lane<4>& d, const Lane<4>& x, int act, float c) { f4_mask(d.a, x.a, act, c); }
__device__ __forceinline__ void lane_mask(Lane<8>& d, const Lane<8>& x, int act, float c) { f4_mask(d.a, x.a, act, c); f4_mask(d.b, x.b, act, c); }

__device__ __forceinline__ void f4_activate(float4& v, int act, float c) {
    // one branch for the four (the activation is the same for the whole launch), so that the clamped-ReLU path does not
    // evaluate the sigmoid's special-function instructions only to discard them
    if (act == ACT_SIGMOID) {
        v.x = activate(v.x, ACT_SIGMOID, c); v.y = activate(v.y, ACT_SIGMOID, c); v.z = activate(v.z, ACT_SIGMOID, c); v.w = activate(v.w, ACT_SIGMOID, c);
    } else {
        v.x = clampf(v.x, c); v.y = clampf(v.y, c); v.z = clampf(v.z, c); v.w = clampf(v.w, c);
    }
}
__device__ __forceinline__ void lane_activate(Lane<4>& v, int act, float c) { f4_activate(v.a, act, c); }
__device__ __forceinline__ void lane_activate(Lane<8>& v, int act, float c) { f4_activate(v.a, act, c); f4_activate(v.b, act, c); }

__device__ __forceinline__ float lane_sum(const Lane<4>& v) { return v.a.x + v.a.y + v.a.z + v.a.w; }
__device__ __forceinline__ float lane_sum(const Lane<8>& v) { return (v.a.x + v.a.y + v.a.z + v.a.w) + (v.b.x + v.b.y + v.b.z + v.b.w); }

// acc += that of the lane whose number differs in bit(s) o; all lanes of the warp
__device__ __forceinline__ void f4_join(float4& v, int o) {
    v.x += __shfl_xor_sync(0xffffffffu, v.x, o); v.y += __shfl_xor_sync(0xffffffffu, v.y, o);
    v.z += __shfl_xor_sync(0xffffffffu, v.z, o); v.w += __shfl_xor_sync(0xffffffffu, v.w, o);
}
__device__ __forceinline__ void lane_join(Lane<4>& v, int o) { f4_join(v.a, o); }
__device__ __forceinline__ void lane_join(Lane<8>& v, int o) { f4_join(v.a, o); f4_join(v.b, o); }

__device__ __forceinline__ bool f4_any(const float4& v) { return !(v.x == 0.0f && v.y == 0.0f && v.z == 0.0f && v.w == 0.0f); }
__device__ __forceinline__ bool lane_any(const Lane<4>& v) { return f4_any(v.a); }
__device__ __forceinline__ bool lane_any(const Lane<8>& v) { return f4_any(v.a) || f4_any(v.b); }

__device__ __forceinline__ unsigned f4_nonzero_bits(const float4& v) {
    return (v.x != 0.0f ? 1u : 0u) | (v.y != 0.0f ? 2u : 0u) | (v.z != 0.0f ? 4u : 0u) | (v.w != 0.0f ? 8u : 0u);
}
__device__ __forceinline__ unsigned lane_nonzero_bits(const Lane<4>& v) { return f4_nonzero_bits(v.a); }
__device__ __forceinline__ unsigned lane_nonzero_bits(const Lane<8>& v) { return f4_nonzero_bits(v.a) | (f4_nonzero_bits(v.b) << 4); }

// S[row,:] += w * d[:] with 128-bit vector reductions
__device__ __forceinline__ void lane_red_add(float* p, float w, const Lane<4>& d) {
    red_add_f4(p, make_float4(w * d.a.x, w * d.a.y, w * d.a.z, w * d.a.w));
}
__device__ __forceinline__ void lane_red_add(float* p, float w, const Lane<8>& d) {
    red_add_f4(p, make_float4(w * d.a.x, w * d.a.y, w * d.a.z, w * d.a.w));
    red_add_f4(p + 4, make_float4(w * d.b.x, w * d.b.y, w * d.b.z, w * d.b.w));
}

template <int G>
__device__ __forceinline__ unsigned group_mask(int grp) {
    return (G == 32) ? 0xffffffffu : (((1u << G) - 1u) << (grp * G));
}

// sum over the G lanes of a row group; `gmask` names exactly those lanes
template <int G>
__device__ __forceinline__ float group_sum(float v, unsigned gmask) {
#pragma unroll
    for (int o = G / 2; o > 0; o >>= 1) v += __shfl_xor_sync(gmask, v, o);
    return v;
}

// The G lanes of a group hold partial sums p0..p3 for the four entries of a chunk.  On return
//   G >= 4: p0 = full sum of entry sub / (G / 4)      (three, four, five shuffles for 4, 8, 16 lanes instead of eight, twelve, sixteen; with the
//   halving only at the last two distances it took 3, 7 and 11: backward 13.66 -> 13.32 us a layer of 16384 neurons and 64 inputs,
//   12.3 -> 11.6 of 6007 and 128)
//   G == 2: p0, p1 = full sums of entries 2*sub, 2*sub+1
//   G == 1: nothing to do.
// The additions pair the same lanes whatever entry a lane ends up owning, so the result does not depend
// on the position of an entry inside its chunk.
template <int G>
__device__ __forceinline__ void chunk_sums(float& p0, float& p1, float& p2, float& p3, int sub, unsigned gmask) {
    if (G >= 4) {
        // halve the number of sums a lane holds at the widest distances, then add up the one that is left
        const bool hi = (sub & (G / 2)) != 0;
        const float s0 = hi ? p0 : p2, s1 = hi ? p1 : p3;
        float k0 = hi ? p2 : p0, k1 = hi ? p3 : p1;
        k0 += __shfl_xor_sync(gmask, s0, G / 2);
        k1 += __shfl_xor_sync(gmask, s1, G / 2);
        const bool odd = (sub & (G / 4)) != 0;
        const float s = odd ? k0 : k1;
        float k = odd ? k1 : k0;
        k += __shfl_xor_sync(gmask, s, G / 4);
#pragma unroll
        for (int o = G / 8; o > 0; o >>= 1) k += __shfl_xor_sync(gmask, k, o);
        p0 = k;
    } else if (G == 2) {
        const bool odd = (sub & 1) != 0;
        const float s0 = odd ? p0 : p2, s1 = odd ? p1 : p3;
        float k0 = odd ? p2 : p0, k1 = odd ? p3 : p1;
        k0 += __shfl_xor_sync(gmask, s0, 1);
        k1 += __shfl_xor_sync(gmask, s1, 1);
        p0 = k0; p1 = k1;
    }
}

// Applies the update w <- w - step*g to the entries of one chunk this lane owns after chunk_sums and
// stores them (entries at positions >= len are padding and stay untouched).  `lim` = len - (first entry this
// lane owns in a chunk), so that "entry stored" is q0 < lim.  DBG: also record the gradient G = g / B.
template <int G, bool DBG>
__device__ __forceinline__ void chunk_update(float* vp, float* gp, const float4& w, float p0, float p1, float p2, float p3,
                                             int sub, int q0, int lim, float step, float inv_b) {
    if (G >= 4) {
        constexpr int SHARE = G >= 4 ? G / 4 : 1;      // lanes that hold the same sum
        const int own = sub / SHARE;
        const float wo = (own & 2) ? ((own & 1) ? w.w : w.z) : ((own & 1) ? w.y : w.x);
        const float nw = __fmaf_rn(-step, p0, wo);
        if ((G == 4 || sub % SHARE == 0) && q0 < lim) {
            vp[own] = nw;
            if (DBG) gp[own] = p0 * inv_b;
        }
    } else if (G == 2) {
        const float wa = sub ? w.z : w.x, wb = sub ? w.w : w.y;
        const int m = 2 * sub;
        const float n0 = __fmaf_rn(-step, p0, wa), n1 = __fmaf_rn(-step, p1, wb);
        if (q0 + 1 < lim) *reinterpret_cast<float2*>(vp + m) = make_float2(n0, n1);      // both entries stored: one 8-byte store
        else if (q0 < lim) vp[m] = n0;
        if (DBG) {
            if (q0 < lim) gp[m] = p0 * inv_b;
            if (q0 + 1 < lim) gp[m + 1] = p1 * inv_b;
        }
    } else {
        const float4 nw = make_float4(__fmaf_rn(-step, p0, w.x), __fmaf_rn(-step, p1, w.y), __fmaf_rn(-step, p2, w.z), __fmaf_rn(-step, p3, w.w));
        if (q0 + 3 < lim) st_f4(vp, nw);      // a whole chunk: one 16-byte store
        else {
            if (q0 + 0 < lim) vp[0] = nw.x;
            if (q0 + 1 < lim) vp[1] = nw.y;
            if (q0 + 2 < lim) vp[2] = nw.z;
        }
        if (DBG) {
            if (q0 + 0 < lim) gp[0] = p0 * inv_b;
            if (q0 + 1 < lim) gp[1] = p1 * inv_b;
            if (q0 + 2 < lim) gp[2] = p2 * inv_b;
            if (q0 + 3 < lim) gp[3] = p3 * inv_b;
        }
    }
}

// ---------------------------------------------------------------------------------------------
// x0 [cnt][n] (input-major, as the caller passes it)  ->  tile [n][ld], zero-padded for b >= cnt.
// Block of 256 threads: 32 inputs x 128 neurons, 16-byte accesses on both sides (where n and the caller's pointer allow it), 16
// KB on their way per block; grid (ceil(n/128), ceil(cols/32)) where cols = padded columns to fill, a multiple of 4.
// With 4-byte accesses and 32 x 32 tiles 65536 x 1024 floats took 213 us in and 178 us out; HBM needs 83.
// row_map (or NULL): tile row of input neuron i, for nets whose input neurons were renumbered at set-up.
constexpr int TRANSPOSE_ROWS = 128, TRANSPOSE_PITCH = 33;
__device__ __forceinline__ void transpose_in(const float* __restrict__ src, float* __restrict__ dst, int n, int cnt, int cols, int ld,
                                             const int* __restrict__ row_map) {
    __shared__ float t[TRANSPOSE_ROWS * TRANSPOSE_PITCH];      // [neuron][input]
    const int i0 = blockIdx.x * TRANSPOSE_ROWS, b0 = blockIdx.y * 32;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, i = i0 + lane * 4;
    const bool wide = (n & 3) == 0 && (reinterpret_cast<unsigned long long>(src) & 15u) == 0;
    float4 v[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const int b = b0 + warp + 8 * j;
        v[j] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (b < cnt) {
            const float* p = src + (size_t)b * n + i;
            if (wide) { if (i < n) v[j] = __ldcs(reinterpret_cast<const float4*>(p)); }
            else {
                if (i + 0 < n) v[j].x = __ldcs(p);
                if (i + 1 < n) v[j].y = __ldcs(p + 1);
                if (i + 2 < n) v[j].z = __ldcs(p + 2);
                if (i + 3 < n) v[j].w = __ldcs(p + 3);
            }
        }
    }
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        float* s = t + lane * 4 * TRANSPOSE_PITCH + warp + 8 * j;
        s[0] = v[j].x; s[TRANSPOSE_PITCH] = v[j].y; s[2 * TRANSPOSE_PITCH] = v[j].z; s[3 * TRANSPOSE_PITCH] = v[j].w;
    }
    __syncthreads();
    const int quad = threadIdx.x & 7;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const int r = (threadIdx.x >> 3) + 32 * j;
        if (i0 + r < n && b0 + quad * 4 < cols) {
            const float* s = t + r * TRANSPOSE_PITCH + quad * 4;
            st_f4(dst + (size_t)(row_map ? row_map[i0 + r] : i0 + r) * ld + b0 + quad * 4, make_float4(s[0], s[1], s[2], s[3]));
        }
    }
}

__global__ void __launch_bounds__(256)
transpose_in_kernel(const float* __restrict__ src, float* __restrict__ dst, int n, int cnt, int cols, int ld, const int* __restrict__ row_map) {
    transpose_in(src, dst, n, cnt, cols, ld, row_map);
}

// tile [n][ld] -> y [cnt][n]; the same blocks
__global__ void __launch_bounds__(256)
transpose_out_kernel(const float* __restrict__ src, float* __restrict__ dst, int n, int cnt, int ld) {
    __shared__ float t[TRANSPOSE_ROWS * TRANSPOSE_PITCH];      // [neuron][input]
    const int i0 = blockIdx.x * TRANSPOSE_ROWS, b0 = blockIdx.y * 32;
    const int quad = threadIdx.x & 7;
    float4 v[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const int r = (threadIdx.x >> 3) + 32 * j;
        v[j] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (i0 + r < n && b0 + quad * 4 < ld) v[j] = ld_f4(src + (size_t)(i0 + r) * ld + b0 + quad * 4);      // ld a multiple of 4
    }
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        float* s = t + ((threadIdx.x >> 3) + 32 * j) * TRANSPOSE_PITCH + quad * 4;
        s[0] = v[j].x; s[1] = v[j].y; s[2] = v[j].z; s[3] = v[j].w;
    }
    __syncthreads();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, i = i0 + lane * 4;
    const bool wide = (n & 3) == 0 && (reinterpret_cast<unsigned long long>(dst) & 15u) == 0;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const int b = b0 + warp + 8 * j;
        if (b < cnt) {
            const float* s = t + lane * 4 * TRANSPOSE_PITCH + warp + 8 * j;
            float* p = dst + (size_t)b * n + i;
            if (wide) { if (i < n) __stcs(reinterpret_cast<float4*>(p), make_float4(s[0], s[TRANSPOSE_PITCH], s[2 * TRANSPOSE_PITCH], s[3 * TRANSPOSE_PITCH])); }
            else {
                if (i + 0 < n) __stcs(p, s[0]);
                if (i + 1 < n) __stcs(p + 1, s[TRANSPOSE_PITCH]);
                if (i + 2 < n) __stcs(p + 2, s[2 * TRANSPOSE_PITCH]);
                if (i + 3 < n) __stcs(p + 3, s[3 * TRANSPOSE_PITCH]);
            }
        }
    }
}

// Start of a train step in one launch: the input tile (blockIdx.z = 0), the target tile (1), and the step's parameters.  sp_batch
// (or NULL): the averaged form, whose backward chain runs on a single vector (sp) while its means are over the batch (sp_batch).
__global__ void __launch_bounds__(256)
start_step_kernel(const float* __restrict__ x0, float* __restrict__ x_tile, const float* __restrict__ target, float* __restrict__ y_tile, int n, int batch,
                  int ld, const int* __restrict__ row_map, StepParams* sp, StepParams* sp_batch, float eta, double* loss) {
    if (blockIdx.x == 0 && blockIdx.y == 0 && blockIdx.z == 0 && threadIdx.x == 0) {
        const int b = sp_batch ? 1 : batch;
        sp->eta = eta; sp->inv_b = 1.0f / (float)b; sp->batch = b; sp->pad = 0;
        if (sp_batch) { sp_batch->eta = eta; sp_batch->inv_b = 1.0f / (float)batch; sp_batch->batch = batch; sp_batch->pad = 0; }
        *loss = 0.0;
    }
    if (blockIdx.z == 0) transpose_in(x0, x_tile, n, batch, ld, ld, row_map);
    else transpose_in(target, y_tile, n, batch, ld, ld, nullptr);
}

// ---------------------------------------------------------------------------------------------
// Forward layer on plain CSR arrays (feedforward equation).  Used only where the stored entries
// belong to the caller and cannot be re-laid out (sdnn_infer_noalloc).
// The arrays are the caller's and were never validated on the host: a column index outside [0, n) is not followed
// (its entry contributes nothing) and is counted in *bad_columns, which the host can read afterwards.
// G lanes hold V inputs each, and S groups of G lanes share a row: group s takes STEP entries of every STEP * S, and the groups' sums meet in
// shuffles.  Rows start anywhere, so the lanes of a group fetch the entries of a step (each lane OWN of
// them side by side, one step ahead; as vectors where the row starts at a multiple of four), check their columns once and hand them
// round by shuffles: STEP gathers of every group are in flight whatever the row's alignment (rows of 8 .. 56 entries, 4096
// neurons, 100 inputs: 14.7 -> 8.5 us per layer, where rows off a multiple of four had taken their entries one at a time).
template <int G, int V, int STEP, int S>
__global__ void __launch_bounds__(256)
forward_csr_kernel(const int* __restrict__ row_ptr, const int* __restrict__ col, const float* __restrict__ val,
                   const float* __restrict__ bias, const float* __restrict__ xin, float* __restrict__ xout,
                   int n, int ld, int last, float clamp, unsigned long long* __restrict__ bad_columns) {
    constexpr int RPW = 32 / (G * S), OWN = (STEP + G - 1) / G;      // entries of a step that a lane fetches (G > STEP: only the first STEP lanes do)
    const int lane = threadIdx.x & 31;
    const int sub = lane % G, lead = lane - sub, part = lane / G % S;
    const int row = (blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5)) * RPW + lane / (G * S);
    int p = 0, e = 0;
    float b = 0.0f;
    if (row < n) { p = row_ptr[row]; e = row_ptr[row + 1]; if (part == 0) b = bias[row]; }
    // the rows of a warp take as many steps as its longest: the shuffles want all lanes
    int steps = (e - p + STEP * S - 1) / (STEP * S);
#pragma unroll
    for (int o = G * S; o < 32; o <<= 1) steps = max(steps, __shfl_xor_sync(0xffffffffu, steps, o));
    const bool aligned = (p & 3) == 0;
    p += part * STEP;
    const int boff = blockIdx.y * (V * G) + sub * V;
    const float* xg = xin + min(boff, last);      // lanes of nothing but padding gather what the last lane with inputs does (no sector more)
    const unsigned pitch = (unsigned)ld * 4u;
    unsigned bad = 0;
    int c[OWN];
    float w[OWN];
    auto fetch = [&](int at) {
        const int first = at + sub * OWN;
        if (OWN >= 4 && aligned && first + OWN <= e) {
#pragma unroll
            for (int i = 0; i + 3 < OWN; i += 4) {
                const int4 cv = __ldg(reinterpret_cast<const int4*>(col + first + i));
                const float4 wv = __ldg(reinterpret_cast<const float4*>(val + first + i));
                c[i] = cv.x; c[i + 1] = cv.y; c[i + 2] = cv.z; c[i + 3] = cv.w;
                w[i] = wv.x; w[i + 1] = wv.y; w[i + 2] = wv.z; w[i + 3] = wv.w;
            }
        } else {
#pragma unroll
            for (int i = 0; i < OWN; ++i) {
                const bool on = first + i < e && sub * OWN < STEP;
                c[i] = on ? __ldg(col + first + i) : 0;
                w[i] = on ? __ldg(val + first + i) : 0.0f;
            }
        }
#pragma unroll
        for (int i = 0; i < OWN; ++i)
            if ((unsigned)c[i] >= (unsigned)n) { ++bad; c[i] = 0; w[i] = 0.0f; }      // not followed, counted once
    };
    fetch(p);
    grid_dependency_wait();
    grid_launch_dependents();
    Lane<V> acc;
    lane_fill(acc, b);
    for (int t = 0; t < steps; ++t, p += STEP * S) {
        Lane<V> x[STEP];
        float ww[STEP];
#pragma unroll
        for (int j = 0; j < STEP; ++j) {
            const int cc = __shfl_sync(0xffffffffu, c[j % OWN], lead + j / OWN);
            ww[j] = __shfl_sync(0xffffffffu, w[j % OWN], lead + j / OWN);
            if (p + j < e) lane_gather(x[j], tile_row(xg, cc, pitch)); else lane_fill(x[j], 0.0f);
        }
        fetch(p + STEP * S);
#pragma unroll
        for (int j = 0; j < STEP; ++j) if (p + j < e) lane_fma(ww[j], x[j], acc);
    }
#pragma unroll
    for (int o = G; o < G * S; o <<= 1) lane_join(acc, o);
    if (bad) atomicAdd(bad_columns, (unsigned long long)bad);
    if (row < n && part == 0) {
        lane_activate(acc, ACT_CLAMPED_RELU, clamp);
        lane_store(tile_row(xout + boff, row, pitch), acc);
    }
}

// ---------------------------------------------------------------------------------------------
// Helpers of the layer kernels' software pipeline.  A step handles CPS chunks (4*CPS entries) of a row, all of
// whose gathers are in flight together; slices are padded to a multiple of 8 entries per row, so a step of
// one or two chunks never needs a guard.  All the rows of a slice run through the slice's padded width
// (padding has index 0 and value 0), which keeps the lanes of a warp converged.  The indices of a step are
// loaded one step ahead (while the previous step's gathers are in flight, also across the boundary between
// two units), so that a step costs one memory round trip, not two dependent ones.
// The four indices of one chunk of one row as they are stored: four 32-bit words, or (I16: nets of at most 65536
// neurons) two words holding four 16-bit indices.  load_idx4 does not touch what it loads, so that the loads of several
// chunks leave back to back (unpacking at the load would make every load wait for its own data before the next one is
// issued); idx_unpack turns a chunk into four indices where they are used.
template <bool I16> struct IdxChunk;
template <> struct IdxChunk<false> { int4 v; };
template <> struct IdxChunk<true> { uint2 v; };
__device__ __forceinline__ void idx_zero(IdxChunk<false>& c) { c.v = make_int4(0, 0, 0, 0); }
__device__ __forceinline__ void idx_zero(IdxChunk<true>& c) { c.v = make_uint2(0u, 0u); }
// `at`: element offset of the chunk in the index array, a multiple of 4
__device__ __forceinline__ void load_idx4(IdxChunk<false>& c, const Sliced& m, int at) {
    c.v = __ldcs(reinterpret_cast<const int4*>(m.idx + at));
}
__device__ __forceinline__ void load_idx4(IdxChunk<true>& c, const Sliced& m, int at) {
    c.v = __ldcs(reinterpret_cast<const uint2*>(reinterpret_cast<const unsigned short*>(m.idx) + at));
}
__device__ __forceinline__ int4 idx_unpack(const IdxChunk<false>& c) { return c.v; }
__device__ __forceinline__ int4 idx_unpack(const IdxChunk<true>& c) {
    return make_int4((int)(c.v.x & 0xffffu), (int)(c.v.x >> 16), (int)(c.v.y & 0xffffu), (int)(c.v.y >> 16));
}
__device__ __forceinline__ int load_idx1(const Sliced& m, int at) {
    return m.idx16 ? (int)reinterpret_cast<const unsigned short*>(m.idx)[at] : m.idx[at];
}
template <int CPS, bool I16>
__device__ __forceinline__ void load_idx(IdxChunk<I16> (&c)[CPS], const Sliced& m, int at) {
#pragma unroll
    for (int i = 0; i < CPS; ++i) load_idx4(c[i], m, at + CHUNK_ROW * i);
}

// asks for the slices that hold the rows of unit `u` (rpw consecutive rows) to be brought into L2
__device__ __forceinline__ void prefetch_unit(const Sliced& m, int u, int rpw, int n, int units_per_slice) {
    const int r0 = u * rpw;
    if (units_per_slice > 1 && (r0 & (SLICE - 1)) != 0) return;      // units narrower than a slice: the first one asks for the whole slice
    const int s0 = r0 / SLICE, s1 = min((n + SLICE - 1) / SLICE, (r0 + rpw - 1) / SLICE + 1);
    const int lo = m.slice_off[s0], hi = m.slice_off[s1];
    if (hi > lo) {
        if (m.idx16) prefetch_l2(reinterpret_cast<const unsigned short*>(m.idx) + lo, (unsigned)(hi - lo) * 2u);
        else prefetch_l2(m.idx + lo, (unsigned)(hi - lo) * 4u);
        prefetch_l2(m.val + lo, (unsigned)(hi - lo) * 4u);
    }
}

#define SDNN_GATHER_CHUNK_SEL(SEL, X, I, C, P, PITCH)                                                     \
    { const int4 cu_ = idx_unpack(C);                                                                     \
      lane_gather_sel<SEL>(X[4 * (I) + 0], tile_row(P, cu_.x, PITCH)); lane_gather_sel<SEL>(X[4 * (I) + 1], tile_row(P, cu_.y, PITCH)); \
      lane_gather_sel<SEL>(X[4 * (I) + 2], tile_row(P, cu_.z, PITCH)); lane_gather_sel<SEL>(X[4 * (I) + 3], tile_row(P, cu_.w, PITCH)); }
#define SDNN_GATHER_CHUNK(X, I, C, P, PITCH)                                                              \
    { const int4 cu_ = idx_unpack(C);                                                                     \
      lane_gather(X[4 * (I) + 0], tile_row(P, cu_.x, PITCH)); lane_gather(X[4 * (I) + 1], tile_row(P, cu_.y, PITCH)); \
      lane_gather(X[4 * (I) + 2], tile_row(P, cu_.z, PITCH)); lane_gather(X[4 * (I) + 3], tile_row(P, cu_.w, PITCH)); }

// Position of a group's item (matrix row, or position in the transposed copy) in unit U of matrix M: BASE =
// element offset of its first chunk, NCH = chunks of its slice (even), ITEM = n for groups beyond the matrix
// (they run through the padding rows of the last slice like everyone else and store nothing).
#define SDNN_UNIT_SHAPE(M, U, NUNITS, ITEM, BASE, NCH)                                        \
    ITEM = (U) * RPW + grp; BASE = 0; NCH = 0;                                                \
    if ((U) < (NUNITS) && (ITEM / SLICE) < ((n + SLICE - 1) / SLICE)) {                       \
        const int so_ = M.slice_off[ITEM / SLICE];                                            \
        BASE = so_ + (ITEM % SLICE) * 4; NCH = (M.slice_off[ITEM / SLICE + 1] - so_) / CHUNK_ROW; \
    }                                                                                         \
    if (ITEM >= n) ITEM = n;

// ---------------------------------------------------------------------------------------------
// Forward layer (feedforward equation): Xout[i,:] = clamp(bias[i] + sum_q val[i,q] * Xin[idx[i,q],:]).
// Persistent grid: a warp takes units (32/G consecutive rows) in a grid-stride loop, or (span > 0) within its CTA's
// run of `span` consecutive units.  One group of G lanes
// per row (SHARE: 2^ls groups, whose sums meet at the row's end); each lane accumulates V batch entries with fp32 FMAs in stored order: ascending
// columns, or, in the copies that stand in for whole networks (resident_reorder_kernel), the order in which those read a row's entries.
// While it works on a unit a warp asks for the entries of its next unit to be brought into L2.
// CG: the gathers go past L1 (64-byte rows of a layer without padding entries).
// SPAN: a CTA takes a run of `span` consecutive units instead of walking the units in a grid-wide stride.
// last: offset of the last lane that holds inputs.  Lanes of nothing but padding gather what that lane gathers (what they store is
// multiplied by the zeros of delta's padding or never read), which adds no sector to a request: rows wider than 64 bytes cost by
// their bytes (40000 neurons, 8 layers, 90 inputs: 319 -> 299 us).
// TRACK (dropping dead inputs): one grid for all chunks, whose warps walk the units of the chunks that still hold live inputs
// (*ncols_dev of them), so that the whole device works on what is left; the columns that stay live are marked in live_flags.  SHARE: 2^ls groups of
// lanes share a row, as in forward_split_kernel, which runs the same layers when nothing is dropped; an instantiation of its own, as a
// number of rows per unit that is known only at run time costs every unit (us for 12 layers, with / without: 20000 neurons, 30 inputs
// 175 / 160; 8000, 257 inputs of which a third survive 258 / 229; 3500, 257 inputs that all do 220 / 204).
// In launches of more than LIVE_WARPS warps the marks of a CTA's rows meet in shared memory and a CTA stores each once: every warp's storing the same few
// words on its own is what such a launch ends with (us a layer, 60 inputs: 2048 neurons 8.7 -> 6.9, 1465 7.15 -> 6.15; 8000 neurons, 257 inputs
// 35 -> 25), while the barrier costs a smaller one 0.3 us (700 neurons, 8 inputs, 88 warps: 4.6, with it 5.0; 2048, 16 inputs, 512: 4.7, 5.0; 1024, 60 inputs, 1024: 5.8,
// 5.6).  Columns beyond LIVE_COLS are marked by their warps.
constexpr int LIVE_WARPS = 768;
constexpr int LIVE_COLS = 4096;
template <int G, int V, int CPS, bool I16, bool CG = false, bool SPAN = false, bool TRACK = false, bool SHARE = false>
__global__ void __launch_bounds__(256, CPS > 2 ? 1 : 2)
forward_kernel(Sliced m, const float* __restrict__ bias, const float* __restrict__ xin, float* __restrict__ xout,
               int n, int ld, float clamp, int act, int pdl, const int* __restrict__ ncols_dev, int* __restrict__ live_flags, int span, int last, int ls) {
    constexpr int LOG_GROUPS = G == 1 ? 5 : G == 2 ? 4 : G == 4 ? 3 : G == 8 ? 2 : G == 16 ? 1 : 0;
    const int log_rows = LOG_GROUPS - (SHARE ? ls : 0), RPW = 1 << log_rows;
    const int UPS = (RPW >= SLICE) ? 1 : SLICE >> log_rows;      // units per slice
    const int lane = threadIdx.x & 31;
    const int sub = lane % G, grp = lane / G >> (SHARE ? ls : 0);
    const int part = SHARE ? (lane / G) & ((1 << ls) - 1) : 0, hop = SHARE ? CPS << ls : CPS, skip = part * CPS;      // this group's steps of its row
    const int wpb = blockDim.x >> 5;
    const int all_units = (n + RPW - 1) >> log_rows;
    const int nunits = SPAN ? min(all_units, ((int)blockIdx.x + 1) * span) : all_units;
    const int stride = SPAN ? wpb : gridDim.x * wpb;
    int boff = (TRACK ? 0 : blockIdx.y * (V * G)) + sub * V;
    const unsigned pitch = (unsigned)ld * 4u;
    const float* __restrict__ val = m.val;
    __shared__ unsigned s_live[TRACK ? LIVE_COLS / 32 : 1];      // a bit per column that a row of this CTA keeps alive
    const bool meet = TRACK && stride > LIVE_WARPS;
    if (meet) {
        for (int c = threadIdx.x; c < LIVE_COLS / 32; c += blockDim.x) s_live[c] = 0u;
        __syncthreads();
    }

    int unit = (SPAN ? blockIdx.x * span : blockIdx.x * wpb) + (threadIdx.x >> 5);
    int chunks_left = 0x7fffffff;      // TRACK: chunks from the current one on
#define SDNN_WRAP(U, BOFF, LEFT) if (TRACK && (U) >= nunits) { const int q_ = (U) / nunits; (U) -= q_ * nunits; BOFF += q_ * (V * G); LEFT -= q_; }
    SDNN_WRAP(unit, boff, chunks_left)
    // prologue that does not depend on the previous layer: shape of the first row, its entries on their way to L2
    int row, base, nch;
    SDNN_UNIT_SHAPE(m, unit, nunits, row, base, nch)
    float b = (row < n && part == 0) ? bias[row] : 0.0f;
    int to = (m.out && row < n) ? m.out[row] : row;       // tile row this row writes
    if (unit < nunits && lane == 0) prefetch_unit(m, unit, RPW, n, UPS);
    IdxChunk<I16> c[CPS];
#pragma unroll
    for (int i = 0; i < CPS; ++i) idx_zero(c[i]);
    if (nch > skip) load_idx<CPS, I16>(c, m, base + skip * CHUNK_ROW);
    if (pdl) grid_dependency_wait();
    if (pdl == 2) grid_launch_dependents();
    int live_cols = 0;
    if (TRACK) {
        live_cols = (*ncols_dev + V * G - 1) / (V * G);
        chunks_left += live_cols - 0x7fffffff;
        live_cols *= V * G;
    }
    unsigned live = 0u;       // bit e: column boff + e of some row this lane produced is nonzero

    while (unit < nunits && (!TRACK || chunks_left > 0)) {
        // shape of this group's row in the warp's next unit (used when this unit's last step prefetches across the boundary)
        int nunit = unit + stride, nboff = boff, nleft = chunks_left;
        SDNN_WRAP(nunit, nboff, nleft)
        int nrow, nbase, nnch;
        SDNN_UNIT_SHAPE(m, nunit, nunits, nrow, nbase, nnch)
        const float nb = (nrow < n && part == 0) ? bias[nrow] : 0.0f;
        const int nto = (m.out && nrow < n) ? m.out[nrow] : nrow;
        if (nunit < nunits && lane == 0) prefetch_unit(m, nunit, RPW, n, UPS);

        Lane<V> acc;
        lane_fill(acc, b);
        const float* vp = val + base;
        const float* xg = xin + (TRACK || G <= 2 ? boff : min(boff, last));
        for (int t = skip; t < nch; t += hop) {
            float4 w[CPS];
            Lane<V> x[4 * CPS];
#pragma unroll
            for (int i = 0; i < CPS; ++i) w[i] = __ldcs(reinterpret_cast<const float4*>(vp + (t + i) * CHUNK_ROW));
#pragma unroll
            for (int i = 0; i < CPS; ++i) { SDNN_GATHER_CHUNK_SEL(CG, x, i, c[i], xg, pitch) }
            if (t + hop < nch) load_idx<CPS, I16>(c, m, base + (t + hop) * CHUNK_ROW);
            else if (nnch > skip) load_idx<CPS, I16>(c, m, nbase + skip * CHUNK_ROW);
#pragma unroll
            for (int i = 0; i < CPS; ++i) {
                lane_fma(w[i].x, x[4 * i + 0], acc); lane_fma(w[i].y, x[4 * i + 1], acc);
                lane_fma(w[i].z, x[4 * i + 2], acc); lane_fma(w[i].w, x[4 * i + 3], acc);
            }
        }
        if (nch <= skip && nnch > skip) load_idx<CPS, I16>(c, m, nbase + skip * CHUNK_ROW);      // no step: nothing prefetched across the boundary yet
        if (SHARE) {
            __syncwarp();
            for (int o = G; o < G << ls; o <<= 1) lane_join(acc, o);
        }
        if (row < n && part == 0) {
            lane_activate(acc, act, clamp);
            lane_store(tile_row(xout + boff, to, pitch), acc);
            if (TRACK) live |= lane_nonzero_bits(acc);
        }
        if (TRACK && (nboff != boff || nleft <= 0)) {      // this warp's last unit of the chunk
            if (meet && boff < LIVE_COLS) {
                __syncwarp();
#pragma unroll
                for (int o = G; o < 32; o <<= 1) live |= __shfl_xor_sync(0xffffffffu, live, o);
                if (lane < G && live) atomicOr(&s_live[boff / 32], live << (boff % 32));
            } else {
#pragma unroll
                for (int e = 0; e < V; ++e)
                    if ((live >> e) & 1u) live_flags[boff + e] = 1;      // many lanes may store the same 1
            }
            live = 0u;
        }
        unit = nunit; row = nrow; base = nbase; nch = nnch; b = nb; to = nto;
        if (TRACK) { boff = nboff; chunks_left = nleft; }
    }
#undef SDNN_WRAP
    if (meet) {
        __syncthreads();
        for (int c = threadIdx.x; c < min(live_cols, LIVE_COLS); c += blockDim.x)
            if ((s_live[c / 32] >> (c % 32)) & 1u) live_flags[c] = 1;
    }
    if (pdl == 1) grid_launch_dependents();
}

// ---------------------------------------------------------------------------------------------
// Forward layer with the gathered operand staged in shared memory (layers whose rows were grouped by the columns
// they share, see reorder.h).  The stored rows of such a layer come group by group; the columns of a group are one
// contiguous range of tile rows, its window; every row of a group is padded to the group's longest row (a multiple of
// eight entries; padding: column 0, value 0), so that the place of every entry follows from the group's base without a
// row pointer.  A group's entries are interleaved over slices of 16 rows like those of Sliced:
//     entry q of the group's row r  ->  g_ebase + (r / 16) * 16 k + (q / 4) * 64 + (r % 16) * 4 + q % 4
// Work item = (group, part of its rows, chunk of TC inputs): the CTA copies the window's TC columns into
// shared memory (16-byte cp.async pieces, all in flight at once), then its warps walk the rows: a lane owns one input,
// reads x[col][input] from the window and accumulates in stored order.  The entries of a row (16-bit column within the window, value) travel through a small
// ring in shared memory per warp: pieces of up to 32 entries are fetched with cp.async WINDOW_RING - 1 pieces ahead and
// read back with warp-wide broadcast loads, so that no warp waits for an L2 round trip per row.  The output row goes
// to the tile row `out[row]`: the number the NEXT layer's grouping gave this neuron.  A random row of the window costs
// a shared-memory wavefront instead of an L2 round trip; the window itself is read once per item, contiguously.
struct Windowed {
    const unsigned short* col;    // column of each entry, relative to its group's window
    const float* val;
    const int* out;               // [n] tile row each stored row writes
    const float* bias;            // [n] in stored order
    const int* g_row0;            // [groups + 1] first stored row of each group
    const int* g_c0;              // [groups] first tile row of each group's window
    const int* g_wlen;            // [groups] rows of the window
    const int* g_ebase;           // [groups] offset of the group's first entry (a multiple of 8)
    const int* g_k;               // [groups] entries per (padded) row of the group, a multiple of 8
    int groups;
};

__device__ __forceinline__ void cp_async16(void* smem_dst, const void* gmem_src) {
    const unsigned d = (unsigned)__cvta_generic_to_shared(smem_dst);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" :: "r"(d), "l"(gmem_src) : "memory");
}
__device__ __forceinline__ void cp_async8(void* smem_dst, const void* gmem_src) {
    const unsigned d = (unsigned)__cvta_generic_to_shared(smem_dst);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" :: "r"(d), "l"(gmem_src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N> __device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" :: "n"(N) : "memory"); }

constexpr int WINDOW_THREADS = 512;
constexpr int WINDOW_RING = 4;                 // pieces of a warp's entry ring
constexpr int WINDOW_PIECE_BYTES = 192;        // 32 entries: 64 bytes of columns, 128 bytes of values
constexpr int WINDOW_RING_BYTES = (WINDOW_THREADS / 32) * WINDOW_RING * WINDOW_PIECE_BYTES;

template <int TC>
__global__ void __launch_bounds__(WINDOW_THREADS, 1)
forward_window_kernel(Windowed m, const float* __restrict__ xin, float* __restrict__ xout, int ld, int chunks, int splits,
                      float clamp, int act, int pdl) {
    extern __shared__ __align__(128) unsigned char window_smem[];
    constexpr int PPR = TC / 4;                           // 16-byte pieces per window row
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
    unsigned char* ring = window_smem + warp * (WINDOW_RING * WINDOW_PIECE_BYTES);
    float* window = reinterpret_cast<float*>(window_smem + WINDOW_RING_BYTES);      // [wlen][TC]
    const int b = min(lane, TC - 1);                      // lanes beyond the chunk repeat its last input and store nothing
    if (pdl) grid_dependency_wait();
    if (pdl == 2) grid_launch_dependents();
    const int per_group = chunks * splits;
    const int items = m.groups * per_group;
    for (int item = blockIdx.x; item < items; item += gridDim.x) {
        const int g = item / per_group, rest = item - g * per_group;
        const int split = rest / chunks, t0 = (rest - split * chunks) * TC;
        const int c0 = m.g_c0[g], wlen = m.g_wlen[g], k = m.g_k[g];
        const int g0 = m.g_row0[g], per_split = (m.g_row0[g + 1] - g0 + splits - 1) / splits;
        const int r0 = g0 + split * per_split + warp, r1 = min(m.g_row0[g + 1], g0 + (split + 1) * per_split);
        const unsigned short* gcol = m.col + m.g_ebase[g];
        const float* gval = m.val + m.g_ebase[g];
        const int ppr = (k + 31) >> 5;                    // pieces per row
        const int my_rows = r0 < r1 ? (r1 - r0 + nwarps - 1) / nwarps : 0;
        const int pieces = my_rows * ppr;
        // piece i of this warp: row r0 + (i / ppr) * nwarps, entries (i % ppr) * 32 .. of that row
        auto fetch = [&](int i) {
            if (i < pieces) {
                const int row = r0 + (i / ppr) * nwarps, t = (i % ppr) << 5;
                const int n = min(32, k - t);             // entries of the piece, a multiple of 8
                const int r = row - g0, q = lane & 7;     // lanes 0 .. 7: four columns each, 8 .. 15: four values
                const size_t at = (size_t)(r & ~(SLICE - 1)) * k + (r & (SLICE - 1)) * 4 + (size_t)((t >> 2) + q) * CHUNK_ROW;
                unsigned char* slot = ring + (i % WINDOW_RING) * WINDOW_PIECE_BYTES;
                if (lane < 16 && q < (n >> 2)) {
                    if (lane < 8) cp_async8(slot + q * 8, gcol + at);
                    else cp_async16(slot + 64 + q * 16, gval + at);
                }
            }
            cp_async_commit();
        };
        __syncthreads();                                  // the previous item's readers are done with the window and the rings
#pragma unroll
        for (int i = 0; i < WINDOW_RING - 1; ++i) fetch(i);
        for (int p = threadIdx.x; p < wlen * PPR; p += blockDim.x) {
            const int r = p / PPR, q = p - r * PPR;
            cp_async16(window + r * TC + q * 4, xin + (size_t)(c0 + r) * ld + t0 + q * 4);
        }
        cp_async_commit();
        cp_async_wait<0>();
        __syncthreads();
        const float* xw = window + b;
        float acc = 0.0f;
        for (int i = 0; i < pieces; ++i) {
            __syncwarp();                                 // every lane has finished reading the slot that is refilled now
            fetch(i + WINDOW_RING - 1);
            cp_async_wait<WINDOW_RING - 1>();             // this lane's share of piece i has landed ...
            __syncwarp();                                 // ... and so has every other lane's
            const int row = r0 + (i / ppr) * nwarps, t = (i % ppr) << 5;
            const int n = min(32, k - t);
            const unsigned char* slot = ring + (i % WINDOW_RING) * WINDOW_PIECE_BYTES;
            if (t == 0) acc = m.bias[row];
            for (int j = 0; j < n; j += 8) {
                const uint4 c = *reinterpret_cast<const uint4*>(slot + j * 2);
                const float4 w0 = *reinterpret_cast<const float4*>(slot + 64 + j * 4);
                const float4 w1 = *reinterpret_cast<const float4*>(slot + 64 + j * 4 + 16);
                const float x0 = xw[(c.x & 0xffffu) * TC], x1 = xw[(c.x >> 16) * TC], x2 = xw[(c.y & 0xffffu) * TC], x3 = xw[(c.y >> 16) * TC];
                const float x4 = xw[(c.z & 0xffffu) * TC], x5 = xw[(c.z >> 16) * TC], x6 = xw[(c.w & 0xffffu) * TC], x7 = xw[(c.w >> 16) * TC];
                acc = fmaf(w0.x, x0, acc); acc = fmaf(w0.y, x1, acc); acc = fmaf(w0.z, x2, acc); acc = fmaf(w0.w, x3, acc);
                acc = fmaf(w1.x, x4, acc); acc = fmaf(w1.y, x5, acc); acc = fmaf(w1.z, x6, acc); acc = fmaf(w1.w, x7, acc);
            }
            if (t + 32 >= k && lane < TC) xout[(size_t)m.out[row] * ld + t0 + lane] = activate(acc, act, clamp);
        }
        if (k == 0 && lane < TC)                          // a group of rows without entries: x = f(b)
            for (int row = r0; row < r1; row += nwarps) xout[(size_t)m.out[row] * ld + t0 + lane] = activate(m.bias[row], act, clamp);
        cp_async_wait<0>();
    }
    if (pdl == 1) grid_launch_dependents();
}

// ---------------------------------------------------------------------------------------------
// The same layer for chunks of 32 inputs with 16 rows side by side in a warp, two lanes a row, 16 inputs a lane: a window row is
// read with four 128-bit loads per lane (a row's two lanes take the halves of one 32-byte sector, the unit the output is stored
// in), and the four rows of a phase (eight lanes) start with different quarters of their
// 128 bytes, so that a phase never meets in a bank.  What bounds the kernel is the shared-memory pipe, one wavefront per stored
// entry and 32 inputs.  A warp's entries come straight from global memory (128 contiguous bytes of columns, 256 of values per four
// entries of 16 rows), two chunks ahead, under the shared-memory reads of the two chunks before them.
// Four rows in a warp and the entries passed through a ring in shared memory cost a fifth of that pipe on top: 65536 neurons in 64
// blocks, six layers of 4096 inputs with the copies in and out 9.83 -> 8.19 ms (8.42 with each lane on its own half of the row); 4096 neurons, 24 layers, 256
// inputs 260 -> 204 us.
constexpr int W32_THREADS = 512;

// acc += w * (the lane's 64 bytes of a window row: every other 16-byte piece), from the piece at `turn` on
__device__ __forceinline__ void window_entry(unsigned row, unsigned turn, float w, float4 (&acc)[4]) {
    float4 x[4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
        asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(x[i].x), "=f"(x[i].y), "=f"(x[i].z), "=f"(x[i].w)
                     : "r"(row + ((turn + i * 32u) & 127u)));
#pragma unroll
    for (int i = 0; i < 4; ++i) f4_fma(w, x[i], acc[i]);
}

__global__ void __launch_bounds__(W32_THREADS, 1)
forward_window32_kernel(Windowed m, const float* __restrict__ xin, float* __restrict__ xout, int ld, int chunks, int splits,
                        float clamp, int act, int pdl) {
    extern __shared__ __align__(128) unsigned char window_smem[];                 // [wlen][32] floats
    constexpr int TC = 32, WARPS = W32_THREADS / 32;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int sub = lane & 1, grp = lane >> 1;
    const unsigned turn = 32u * (grp & 3);
    const unsigned xw = (unsigned)__cvta_generic_to_shared(window_smem) + sub * 16u;
    if (pdl) grid_dependency_wait();
    if (pdl == 2) grid_launch_dependents();
    const int per_group = chunks * splits;
    const int items = m.groups * per_group;
    for (int item = blockIdx.x; item < items; item += gridDim.x) {
        const int g = item / per_group, rest = item - g * per_group;
        const int split = rest / chunks, t0 = (rest - split * chunks) * TC;
        const int c0 = m.g_c0[g], wlen = m.g_wlen[g], k = m.g_k[g], nch = k >> 2;
        const int g0 = m.g_row0[g], rows = m.g_row0[g + 1] - g0, slices = (rows + SLICE - 1) / SLICE;
        const int per_split = (slices + splits - 1) / splits;
        const int s1 = min(slices, (split + 1) * per_split);
        int s = split * per_split + warp;                                         // this warp's slice of the group
        const unsigned short* gcol = m.col + m.g_ebase[g] + grp * 4;
        const float* gval = m.val + m.g_ebase[g] + grp * 4;
        uint2 c_a = make_uint2(0u, 0u), c_b = c_a;
        float4 w_a = make_float4(0.f, 0.f, 0.f, 0.f), w_b = w_a;
        float bias = 0.0f;
        int to = 0;
        auto place = [&](int sl) { const int r = min(sl * SLICE + grp, rows - 1); bias = m.bias[g0 + r]; to = m.out[g0 + r]; };
        if (s < s1) {                                                             // first two chunks, bias and place of the first slice
            const size_t at = (size_t)s * SLICE * k;
            if (nch) {
                c_a = __ldg(reinterpret_cast<const uint2*>(gcol + at));
                w_a = __ldg(reinterpret_cast<const float4*>(gval + at));
                c_b = __ldg(reinterpret_cast<const uint2*>(gcol + at + CHUNK_ROW));
                w_b = __ldg(reinterpret_cast<const float4*>(gval + at + CHUNK_ROW));
            }
            place(s);
        }
        __syncthreads();                                                          // the previous item's readers are done with the window
        for (int p = threadIdx.x; p < wlen * (TC / 4); p += W32_THREADS)
            cp_async16(window_smem + p * 16, xin + (size_t)(c0 + (p >> 3)) * ld + t0 + (p & 7) * 4);
        cp_async_commit();
        cp_async_wait<0>();
        __syncthreads();
        for (; s < s1; s += WARPS) {
            const size_t at = (size_t)s * SLICE * k, next = (size_t)(s + WARPS < s1 ? s + WARPS : s) * SLICE * k;
            const float b = bias;
            const int row_to = to;
            const bool stored = s * SLICE + grp < rows;
            if (s + WARPS < s1) place(s + WARPS);
            float4 acc[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) acc[i] = make_float4(0.f, 0.f, 0.f, 0.f);
            // chunk T, held in (c, w): a window row is 128 bytes; then the registers take the chunk two further on, at the end
            // of a slice the first two of the warp's next one
            auto chunk = [&](uint2& c, float4& w, int T) {
                const unsigned a0 = xw + ((c.x & 0xffffu) << 7), a1 = xw + ((c.x >> 16) << 7);
                const unsigned a2 = xw + ((c.y & 0xffffu) << 7), a3 = xw + ((c.y >> 16) << 7);
                const float4 wv = w;
                const size_t q = T + 2 < nch ? at + (size_t)(T + 2) * CHUNK_ROW : next + (size_t)(T & 1) * CHUNK_ROW;
                c = __ldg(reinterpret_cast<const uint2*>(gcol + q));
                w = __ldg(reinterpret_cast<const float4*>(gval + q));
                window_entry(a0, turn, wv.x, acc);
                window_entry(a1, turn, wv.y, acc);
                window_entry(a2, turn, wv.z, acc);
                window_entry(a3, turn, wv.w, acc);
            };
            for (int t = 0; t < nch; t += 2) {                                    // k is a multiple of eight
                chunk(c_a, w_a, t);
                chunk(c_b, w_b, t + 1);
            }
            if (stored) {                                                         // also the rows of a group without entries (k = 0): x = f(b)
                float* dst = xout + (size_t)row_to * ld + t0 + sub * 4;
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    acc[i].x += b; acc[i].y += b; acc[i].z += b; acc[i].w += b;
                    f4_activate(acc[i], act, clamp);
                    st_f4(dst + (((turn + i * 32u) & 127u) >> 2), acc[i]);
                }
            }
        }
    }
    if (pdl == 1) grid_launch_dependents();
}

// ---------------------------------------------------------------------------------------------
// Output gradient (final-layer gradient equation) and loss: delta^L = (x^L - y) (.) f'(x^L) on the valid
// batch columns, 0 on the padding; J = 1/(2B) sum (x^L - y)^2 accumulated in double, one atomic per block.
__global__ void __launch_bounds__(256)
output_gradient_kernel(const float* __restrict__ xl, const float* __restrict__ y, float* __restrict__ delta,
                       int n, int ld, float clamp, int act, const StepParams* __restrict__ sp, double* __restrict__ loss) {
    const int per_row = ld >> 2;
    const long long total = (long long)n * per_row;
    const int nb = sp->batch;
    float sq = 0.0f;
    for (long long v = (long long)blockIdx.x * blockDim.x + threadIdx.x; v < total; v += (long long)gridDim.x * blockDim.x) {
        const int boff = (int)(v % per_row) * 4;
        const float4 x = ld_f4(xl + v * 4), t = ld_f4(y + v * 4);
        float4 e;
        e.x = (boff + 0 < nb) ? x.x - t.x : 0.0f; e.y = (boff + 1 < nb) ? x.y - t.y : 0.0f;
        e.z = (boff + 2 < nb) ? x.z - t.z : 0.0f; e.w = (boff + 3 < nb) ? x.w - t.w : 0.0f;
        sq += e.x * e.x + e.y * e.y + e.z * e.z + e.w * e.w;
        st_f4(delta + v * 4, make_float4(e.x * derivative(x.x, act, clamp), e.y * derivative(x.y, act, clamp),
                                         e.z * derivative(x.z, act, clamp), e.w * derivative(x.w, act, clamp)));
    }
    __shared__ float part[8];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) sq += __shfl_xor_sync(0xffffffffu, sq, o);
    if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = sq;
    __syncthreads();
    if (threadIdx.x == 0) {
        double tot = 0.0;
        for (int q = 0; q < (int)(blockDim.x >> 5); ++q) tot += (double)part[q];
        if (tot != 0.0) atomicAdd(loss, 0.5 * tot * (double)sp->inv_b);
    }
}

// ---------------------------------------------------------------------------------------------
// Minibatch step in the averaged form (Discussion of Section 5: the output gradients of the batch are averaged and ONE vector is
// backpropagated, SpBP running as for a single input).  The single input SpBP then works with is the batch mean of
// each x^k; the two kernels below form those means and the averaged delta^L as tiles of padded width 4 (value in
// column 0, zeros in columns 1..3), which the backward kernels process like a step with B = 1.
//   spb: the real batch (batch = B, inv_b = 1/B); sums run over b = 0..B-1 in that order.
__global__ void __launch_bounds__(256)
batch_mean_kernel(const float* __restrict__ acts, float* __restrict__ mean, long long rows, int ld,
                  const StepParams* __restrict__ spb) {
    const int nb = spb->batch;
    const float inv = spb->inv_b;
    for (long long r = (long long)blockIdx.x * blockDim.x + threadIdx.x; r < rows; r += (long long)gridDim.x * blockDim.x) {
        const float* a = acts + r * ld;
        float s = 0.0f;
        for (int b = 0; b < nb; ++b) s += a[b];
        st_f4(mean + r * 4, make_float4(s * inv, 0.0f, 0.0f, 0.0f));
    }
}

// delta^L = (1/B) sum_b (x^L_b - y_b) (.) f'(x^L_b); J = 1/(2B) sum_b |x^L_b - y_b|^2 as in output_gradient_kernel.
__global__ void __launch_bounds__(256)
output_gradient_averaged_kernel(const float* __restrict__ xl, const float* __restrict__ y, float* __restrict__ delta,
                                int n, int ld, float clamp, int act, const StepParams* __restrict__ spb,
                                double* __restrict__ loss) {
    const int nb = spb->batch;
    float sq = 0.0f;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const float* x = xl + (size_t)i * ld;
        const float* t = y + (size_t)i * ld;
        float acc = 0.0f;
        for (int b = 0; b < nb; ++b) {
            const float e = x[b] - t[b];
            sq = fmaf(e, e, sq);
            acc = fmaf(e, derivative(x[b], act, clamp), acc);
        }
        st_f4(delta + (size_t)i * 4, make_float4(acc * spb->inv_b, 0.0f, 0.0f, 0.0f));
    }
    __shared__ float part[8];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) sq += __shfl_xor_sync(0xffffffffu, sq, o);
    if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = sq;
    __syncthreads();
    if (threadIdx.x == 0) {
        double tot = 0.0;
        for (int q = 0; q < (int)(blockDim.x >> 5); ++q) tot += (double)part[q];
        if (tot != 0.0) atomicAdd(loss, 0.5 * tot * (double)spb->inv_b);
    }
}

// ---------------------------------------------------------------------------------------------
// Backward + update of one layer k (Algorithm 1, loop body), two realisations.
//
// Row units (always): for row i of W^k with delta^k[i,:] in registers, for each stored (i,j):
//       g = sum_b delta^k[i,b] x^{k-1}[j,b]      (masked gradient times B; x^{k-1}[j,:] gathered)
//       W(i,j) = w - (eta/B) g
//   SCATTER (atomics realisation) additionally S_{k-1}[j,:] += w * delta^k[i,:] with 128-bit vector
//   reductions, w being the value BEFORE the update; there delta^k[i,:] = S_k[i,:] (.) f'(x^k[i,:])
//   is formed on the fly and S_k is cleared row by row as it is consumed (FROM_S).
//
// Column units (transposed realisation, MIRROR): for column j of W^k (a row of the transposed copy,
//   which has its own value array kept bit-identical to the row-major one), with x^{k-1}[j,:] in registers:
//       acc  = sum_i w(i,j) delta^k[i,:]            (delta^k[i,:] gathered; w BEFORE the update)
//       g, update of the transposed copy's value: same arithmetic, same bits as the row unit's
//       delta^{k-1}[j,:] = acc (.) f'(x^{k-1}[j,:])
//   No atomics; one gather per stored entry serves both the product and the gradient.
//
// A warp processes its column units (if any) first, then its row units; both only read delta^k and
// x^{k-1}, so they are independent of each other.  The whole minibatch sits in one chunk (ld = V*G <= 128).
// Same software pipeline as the forward kernel; in addition the resident operand of a unit (delta^k row or
// x^{k-1} row) is loaded during the last step of the unit before it.
struct BackwardArgs {
    Sliced rows;              // row-major copy of W^k
    Sliced cols;              // transposed copy (MIRROR)
    float* bias;              // b^k (updated when update_bias)
    const float* xk;          // x^k tile        (FROM_S: derivative mask of delta^k)
    const float* xprev;       // x^{k-1} tile
    float* dk;                // delta^k tile, or S_k when FROM_S (cleared as consumed)
    float* dprev;             // SCATTER: S_{k-1};  MIRROR: delta^{k-1} tile;  else unused
    float* dbg_delta;         // DBG: copy of delta^k (FROM_S only; otherwise dk is the record)
    float* dbg_grad;          // DBG: G^k in the row-major copy's layout
    const StepParams* sp;
    int n;
    float clamp;
    int act;                  // activation (ACT_*)
    int update_bias, skip_dead, pdl;
    int cols_only;            // MIRROR: leave the row units to a separate launch (which may run beside the next layer's column units)
    int alternate;            // column units: see backward_col_units
    const float* warm;        // tile the NEXT backward launch will gather from (x^{k-2}), or NULL: asked into L2 now,
    unsigned warm_bytes;      // because it was written a whole forward pass ago and has left the cache
};

// Column units of the transposed realisation.  (Lanes of nothing but padding gather their zeros: sending them to the last lane with
// inputs, as the forward kernel does, costs registers that this kernel does not have; 16384 neurons: 2 to 3 % faster at 37
// inputs, 1 to 2 % slower at 64.)
template <int G, int V, int CPS, bool I16>
__device__ __forceinline__ void backward_col_units(const Sliced m, const float* __restrict__ xprev, const float* __restrict__ dk,
                                                   float* __restrict__ dprev, int n, float clamp, int act, float step, float inv_b,
                                                   int first, int stride, int pdl, int alternate) {
    constexpr int RPW = 32 / G;
    constexpr int UPS = (RPW >= SLICE) ? 1 : SLICE / RPW;
    constexpr unsigned pitch = 4u * V * G;
    const int lane = threadIdx.x & 31;
    const int sub = lane % G, grp = lane / G;
    const unsigned gmask = (G >= 2) ? 0xffffffffu : group_mask<G>(grp);     // G >= 2: one slice per warp, its lanes stay converged
    const int nunits = (n + RPW - 1) / RPW;
    const int boff = sub * V;
    float* val = m.val;
    const float* dg = dk + boff;

    // The columns come by descending length.  alternate: a warp that takes several units takes them from alternating ends of
    // its rounds (its hops add up to two strides), so that every warp gets long and short columns (two units each, no row units
    // beside them: 13.4 -> 12.8 us per layer at 16384 neurons and 64 inputs; row units fill the tail as well and gain nothing
    // by it).  Tiles of at least 32 inputs only: narrower ones never ask for it, and the registers it takes cost them 0.7 %.
    int u = first, item, base, nch;
    int hop = G > 2 && alternate ? 2 * (stride - first) - 1 : stride;
    SDNN_UNIT_SHAPE(m, u, nunits, item, base, nch)
    if (u < nunits && lane == 0) prefetch_unit(m, u, RPW, n, UPS);
    int len = 0, j = 0;
    if (item < n) { len = m.len[item]; j = m.order[item]; }
    IdxChunk<I16> c[CPS];
#pragma unroll
    for (int i = 0; i < CPS; ++i) idx_zero(c[i]);
    if (nch > 0) load_idx<CPS, I16>(c, m, base);
    Lane<V> xj;
    lane_fill(xj, 0.0f);
    if (item < n) lane_load(xj, tile_row(xprev + boff, j, pitch));
    // everything above is static for the chain of launches (shapes, indices, x^{k-1}); delta^k is what the launch waits for
    if (pdl) grid_dependency_wait();
    if (pdl == 2) grid_launch_dependents();

    while (u < nunits) {
        const int nu = u + hop;
        if (G > 2) hop = 2 * stride - hop;
        int nitem, nbase, nnch, nlen = 0, nj = 0;
        SDNN_UNIT_SHAPE(m, nu, nunits, nitem, nbase, nnch)
        if (nitem < n) { nlen = m.len[nitem]; nj = m.order[nitem]; }
        if (nu < nunits && lane == 0) prefetch_unit(m, nu, RPW, n, UPS);
        Lane<V> nxj, acc;
        lane_fill(nxj, 0.0f);
        lane_fill(acc, 0.0f);
        float* vp = val + base;
        const int lim = len - ((G >= 4) ? sub / (G >= 4 ? G / 4 : 1) : (G == 2) ? 2 * sub : 0);
#define SDNN_COL_NEXT if (nnch > 0) load_idx<CPS, I16>(c, m, nbase); if (nitem < n) lane_load(nxj, tile_row(xprev + boff, nj, pitch));
        for (int t = 0; t < nch; t += CPS) {
            float4 w[CPS];
            Lane<V> d[4 * CPS];
#pragma unroll
            for (int i = 0; i < CPS; ++i) w[i] = __ldcs(reinterpret_cast<const float4*>(vp + (t + i) * CHUNK_ROW));
#pragma unroll
            for (int i = 0; i < CPS; ++i) { SDNN_GATHER_CHUNK(d, i, c[i], dg, pitch) }
            if (t + CPS < nch) { load_idx<CPS, I16>(c, m, base + (t + CPS) * CHUNK_ROW); }
            else { SDNN_COL_NEXT }
#pragma unroll
            for (int i = 0; i < CPS; ++i) {
                lane_fma(w[i].x, d[4 * i + 0], acc); lane_fma(w[i].y, d[4 * i + 1], acc);
                lane_fma(w[i].z, d[4 * i + 2], acc); lane_fma(w[i].w, d[4 * i + 3], acc);
                float p0 = lane_dot(d[4 * i + 0], xj), p1 = lane_dot(d[4 * i + 1], xj), p2 = lane_dot(d[4 * i + 2], xj), p3 = lane_dot(d[4 * i + 3], xj);
                chunk_sums<G>(p0, p1, p2, p3, sub, gmask);
                chunk_update<G, false>(vp + (t + i) * CHUNK_ROW, nullptr, w[i], p0, p1, p2, p3, sub, (t + i) * 4, lim, step, inv_b);
            }
        }
        if (nch == 0) { SDNN_COL_NEXT }
#undef SDNN_COL_NEXT
        if (item < n) {
            lane_mask(acc, xj, act, clamp);
            lane_store(tile_row(dprev + boff, j, pitch), acc);
        }
        u = nu; item = nitem; base = nbase; nch = nnch; len = nlen; j = nj; xj = nxj;
    }
}

// Row units.
template <int G, int V, int CPS, bool I16, bool FROM_S, bool SCATTER, bool DBG>
__device__ __forceinline__ void backward_row_units(const Sliced m, float* __restrict__ bias, const float* __restrict__ xk,
                                                   const float* __restrict__ xprev, float* dk, float* dprev,
                                                   float* __restrict__ dbg_delta, float* __restrict__ dbg_grad, int n, float clamp, int act,
                                                   float step, float inv_b, int update_bias, int skip_dead, int first, int stride) {
    constexpr int RPW = 32 / G;
    constexpr int UPS = (RPW >= SLICE) ? 1 : SLICE / RPW;
    constexpr unsigned pitch = 4u * V * G;
    const int lane = threadIdx.x & 31;
    const int sub = lane % G, grp = lane / G;
    const unsigned gmask1 = group_mask<G>(grp);
    const unsigned gmask = (G >= 2) ? 0xffffffffu : gmask1;
    const int nunits = (n + RPW - 1) / RPW;
    const int boff = sub * V;
    float* val = m.val;
    const float* xg = xprev + boff;
    float* sg = SCATTER ? dprev + boff : nullptr;

    int u = first, item, base, nch;
    SDNN_UNIT_SHAPE(m, u, nunits, item, base, nch)
    if (u < nunits && lane == 0) prefetch_unit(m, u, RPW, n, UPS);
    int len = (item < n) ? m.len[item] : 0;
    IdxChunk<I16> c[CPS];
#pragma unroll
    for (int i = 0; i < CPS; ++i) idx_zero(c[i]);
    if (nch > 0) load_idx<CPS, I16>(c, m, base);
    Lane<V> h0, h1;       // delta^k[i,:] (or S_k[i,:]) and, FROM_S, x^k[i,:]
    lane_fill(h0, 0.0f); lane_fill(h1, 0.0f);
    // tile row of stored row `item`: its neuron's number (the stored rows of a regrouped layer are not in neuron order)
    int lab = (item < n && m.out) ? m.out[item] : item;
    if (item < n) { lane_load(h0, tile_row(dk + boff, lab, pitch)); if (FROM_S) lane_load(h1, tile_row(xk + boff, lab, pitch)); }

    while (u < nunits) {
        const int nu = u + stride;
        int nitem, nbase, nnch;
        SDNN_UNIT_SHAPE(m, nu, nunits, nitem, nbase, nnch)
        const int nlen = (nitem < n) ? m.len[nitem] : 0;
        const int nlab = (nitem < n && m.out) ? m.out[nitem] : nitem;
        if (nu < nunits && lane == 0) prefetch_unit(m, nu, RPW, n, UPS);
        Lane<V> nh0, nh1;
        lane_fill(nh0, 0.0f); lane_fill(nh1, 0.0f);
        Lane<V> d = h0;
        if (item < n) {
            if (FROM_S) {
                Lane<V> z;
                lane_fill(z, 0.0f);
                lane_store(tile_row(dk + boff, lab, pitch), z);
                lane_mask(d, h1, act, clamp);
                if (DBG) lane_store(tile_row(dbg_delta + boff, lab, pitch), d);
            }
            if (update_bias) {       // bias read as one more column of W^k whose input is the constant 1
                const float bg = group_sum<G>(lane_sum(d), gmask1);
                if (sub == 0) bias[item] -= step * bg;
            }
        }
        if (skip_dead) {             // delta^k(i) = 0 for every input of every row of the unit: nothing changes
            if (__ballot_sync(gmask, lane_any(d)) == 0u) nch = 0;
        }
        float* vp = val + base;
        float* gp = DBG ? dbg_grad + base : nullptr;
        const int lim = len - ((G >= 4) ? sub / (G >= 4 ? G / 4 : 1) : (G == 2) ? 2 * sub : 0);
#define SDNN_ROW_NEXT                                                                                    \
        if (nnch > 0) load_idx<CPS, I16>(c, m, nbase);                                                        \
        if (nitem < n) { lane_load(nh0, tile_row(dk + boff, nlab, pitch)); if (FROM_S) lane_load(nh1, tile_row(xk + boff, nlab, pitch)); }
#define SDNN_SCAT(C, W, Q) if ((Q) < len) lane_red_add(tile_row(sg, C, pitch), W, d);
        for (int t = 0; t < nch; t += CPS) {
            float4 w[CPS];
            Lane<V> x[4 * CPS];
#pragma unroll
            for (int i = 0; i < CPS; ++i) w[i] = __ldcs(reinterpret_cast<const float4*>(vp + (t + i) * CHUNK_ROW));
#pragma unroll
            for (int i = 0; i < CPS; ++i) { SDNN_GATHER_CHUNK(x, i, c[i], xg, pitch) }
            if (SCATTER) {       // stored entries only: padding must not touch S
#pragma unroll
                for (int i = 0; i < CPS; ++i) {
                    const int q = 4 * (t + i);
                    const int4 cu = idx_unpack(c[i]);
                    SDNN_SCAT(cu.x, w[i].x, q) SDNN_SCAT(cu.y, w[i].y, q + 1) SDNN_SCAT(cu.z, w[i].z, q + 2) SDNN_SCAT(cu.w, w[i].w, q + 3)
                }
            }
            if (t + CPS < nch) { load_idx<CPS, I16>(c, m, base + (t + CPS) * CHUNK_ROW); }
            else { SDNN_ROW_NEXT }
#pragma unroll
            for (int i = 0; i < CPS; ++i) {
                float p0 = lane_dot(d, x[4 * i + 0]), p1 = lane_dot(d, x[4 * i + 1]), p2 = lane_dot(d, x[4 * i + 2]), p3 = lane_dot(d, x[4 * i + 3]);
                chunk_sums<G>(p0, p1, p2, p3, sub, gmask);
                chunk_update<G, DBG>(vp + (t + i) * CHUNK_ROW, DBG ? gp + (t + i) * CHUNK_ROW : nullptr, w[i], p0, p1, p2, p3, sub,
                                     (t + i) * 4, lim, step, inv_b);
            }
        }
        if (nch == 0) { SDNN_ROW_NEXT }
#undef SDNN_ROW_NEXT
#undef SDNN_SCAT
        u = nu; item = nitem; base = nbase; nch = nnch; len = nlen; h0 = nh0; h1 = nh1; lab = nlab;
    }
}

template <int G, int V, int CPS, bool I16, bool FROM_S, bool SCATTER, bool MIRROR, bool DBG>
__global__ void __launch_bounds__(256, 2)
backward_kernel(const BackwardArgs a) {
    const int wpb = blockDim.x >> 5;
    const int stride = gridDim.x * wpb;
    const int first = blockIdx.x * wpb + (threadIdx.x >> 5);
    if (a.warm && (threadIdx.x & 31) == 0) {      // each warp asks for its share, in pieces of 4 KB
        const unsigned pieces = (a.warm_bytes + 4095u) >> 12;
        for (unsigned q = first; q < pieces; q += stride) {
            const unsigned lo = q << 12, len = min(4096u, a.warm_bytes - lo);
            prefetch_l2(reinterpret_cast<const char*>(a.warm) + lo, len & ~15u);
        }
    }
    // step parameters: written once per step, long before any backward launch
    const float inv_b = a.sp->inv_b;
    const float step = a.sp->eta * inv_b;
    if (MIRROR) backward_col_units<G, V, CPS, I16>(a.cols, a.xprev, a.dk, a.dprev, a.n, a.clamp, a.act, step, inv_b, first, stride, a.pdl, a.alternate);
    else {
        if (a.pdl) grid_dependency_wait();
        if (a.pdl == 2) grid_launch_dependents();
    }
    if (MIRROR && a.cols_only) { if (a.pdl == 1) grid_launch_dependents(); return; }
    backward_row_units<G, V, CPS, I16, FROM_S, SCATTER, DBG>(a.rows, a.bias, a.xk, a.xprev, a.dk, a.dprev, a.dbg_delta, a.dbg_grad, a.n,
                                                        a.clamp, a.act, step, inv_b, a.update_bias, a.skip_dead, first, stride);
    if (a.pdl == 1) grid_launch_dependents();
}

// ---------------------------------------------------------------------------------------------
// Layers that do not fill the device (train steps: see sdnn_plan::split_units; inference: sdnn_plan::split_rows).  A launch of fewer row groups than warps fit is over when its
// longest row is: 7 dependent round trips of 8 gathers for a row of 56 entries, while the short rows' warps have ended and the request
// path idles.  Here the steps of a long row are dealt to 2, 4, .. groups of G lanes of a warp, whose partial sums meet in shuffles, as
// far as all units still fit the device in one round: `units` lists, for every warp, its first row * 8 + log2(groups per row).
// us a layer, as it was / split: 6007 neurons, rows of 8 to 56 entries, 37 inputs: forward 7.17 / 5.12, backward 8.37 / 7.01; 3000 neurons,
// 32 a row, 12 inputs: 3.92 / 2.56, 5.11 / 3.92; 700 neurons, 64 inputs: 3.58 / 2.21, 4.77 / 3.24.
// A warp has one unit and so nothing to ask for ahead of time but what the next launch will read: the entries of its layer, in pieces
// of 4 KB, where a pass over the net walks so much that they are not at hand (sdnn_plan::asks_ahead; a step of 6007 x 56, 37 inputs 691 -> 654
// us, 3000 x 56, 100 inputs 625 -> 596; 700 x 24, 16 inputs, which do not ask, 142 -> 134).
struct NextEntries { const void* idx; const float* val; unsigned idx_bytes, val_bytes; };
__device__ __forceinline__ void ask_for(const void* base, unsigned bytes, unsigned first, unsigned stride) {
    for (unsigned long long lo = (unsigned long long)first << 12; lo < bytes; lo += (unsigned long long)stride << 12)
        prefetch_l2(reinterpret_cast<const char*>(base) + lo, min(4096u, bytes - (unsigned)lo) & ~15u);
}
struct SplitUnit { int row, part, parts; };
// units NULL: every row is split into 2^ls parts
template <int G>
__device__ __forceinline__ SplitUnit split_unit(const unsigned* units, int ls, int u, int nunits, int grp) {
    if (u >= nunits) return SplitUnit{0x7fffffff, 0, 1};
    const unsigned d = units ? units[u] : (unsigned)(u * (32 / G >> ls)) << 3 | (unsigned)ls;
    ls = d & 7u;
    return SplitUnit{(int)(d >> 3) + (grp >> ls), grp & ((1 << ls) - 1), 1 << ls};
}

constexpr int SPLIT_WARPS = 4;      // of a forward CTA
template <int G, bool I16>
__global__ void __launch_bounds__(32 * SPLIT_WARPS, 16 / SPLIT_WARPS)
forward_split_kernel(Sliced m, const unsigned* __restrict__ units, int ls, int nunits, const float* __restrict__ bias, const float* __restrict__ xin,
                     float* __restrict__ xout, int n, int ld, float clamp, int act, int pdl, int last, NextEntries next) {
    constexpr int V = 8, CPS = 2;
    const unsigned pitch = 4u * ld;
    const int lane = threadIdx.x & 31, sub = lane % G;
    if (lane == 0) {
        const unsigned w = blockIdx.x * SPLIT_WARPS + (threadIdx.x >> 5), warps = gridDim.x * SPLIT_WARPS;
        ask_for(next.val, next.val_bytes, w, warps);
        ask_for(next.idx, next.idx_bytes, w, warps);
    }
    const SplitUnit s = split_unit<G>(units, ls, blockIdx.x * SPLIT_WARPS + (threadIdx.x >> 5), nunits, lane / G);
    int nch = 0, base = 0, to = 0;
    float b = 0.0f;
    IdxChunk<I16> c[CPS];
    if (s.row < n) {
        const int so = m.slice_off[s.row / SLICE];
        nch = (m.slice_off[s.row / SLICE + 1] - so) / CHUNK_ROW;
        base = so + (s.row % SLICE) * 4;
        to = m.out ? m.out[s.row] : s.row;
        if (s.part == 0) b = bias[s.row];
        if (s.part * CPS < nch) load_idx<CPS, I16>(c, m, base + s.part * CPS * CHUNK_ROW);
    }
    if (pdl) grid_dependency_wait();
    if (pdl == 2) grid_launch_dependents();
    Lane<V> acc;
    lane_fill(acc, b);
    const float* vp = m.val + base;
    const float* xg = xin + min(sub * V, last);
    for (int t = s.part * CPS; t < nch; t += s.parts * CPS) {
        float4 w[CPS];
        Lane<V> x[4 * CPS];
#pragma unroll
        for (int i = 0; i < CPS; ++i) w[i] = __ldcs(reinterpret_cast<const float4*>(vp + (t + i) * CHUNK_ROW));
#pragma unroll
        for (int i = 0; i < CPS; ++i) { SDNN_GATHER_CHUNK(x, i, c[i], xg, pitch) }
        if (t + s.parts * CPS < nch) load_idx<CPS, I16>(c, m, base + (t + s.parts * CPS) * CHUNK_ROW);
#pragma unroll
        for (int i = 0; i < CPS; ++i) {
            lane_fma(w[i].x, x[4 * i + 0], acc); lane_fma(w[i].y, x[4 * i + 1], acc);
            lane_fma(w[i].z, x[4 * i + 2], acc); lane_fma(w[i].w, x[4 * i + 3], acc);
        }
    }
    __syncwarp();
    for (int o = G; o < G * s.parts; o <<= 1) lane_join(acc, o);
    if (s.row < n && s.part == 0) {
        lane_activate(acc, act, clamp);
        lane_store(tile_row(xout + sub * V, to, pitch), acc);
    }
    if (pdl == 1) grid_launch_dependents();
}

// Column units: as backward_col_units, per entry the same arithmetic.  CTAs of one warp, like the launches they run beside.
template <int G, bool I16>
__global__ void __launch_bounds__(32, 16)
backward_split_kernel(Sliced m, const unsigned* __restrict__ units, int nunits, const float* __restrict__ xprev, const float* __restrict__ dk,
                      float* __restrict__ dprev, int n, float clamp, int act, const StepParams* __restrict__ sp, int pdl,
                      const float* __restrict__ warm, unsigned warm_bytes, NextEntries next) {
    constexpr int V = 8, CPS = 2;
    constexpr unsigned pitch = 4u * V * G;
    const int lane = threadIdx.x, sub = lane % G;
    if (lane == 0) {
        ask_for(next.val, next.val_bytes, blockIdx.x, gridDim.x);
        ask_for(next.idx, next.idx_bytes, blockIdx.x, gridDim.x);
        ask_for(warm, warm_bytes, blockIdx.x, gridDim.x);
    }
    const float inv_b = sp->inv_b, step = sp->eta * inv_b;
    const SplitUnit s = split_unit<G>(units, 0, blockIdx.x, nunits, lane / G);
    int nch = 0, base = 0, len = 0, j = 0;
    IdxChunk<I16> c[CPS];
#pragma unroll
    for (int i = 0; i < CPS; ++i) idx_zero(c[i]);
    Lane<V> xj, acc;
    lane_fill(xj, 0.0f);
    lane_fill(acc, 0.0f);
    if (s.row < n) {
        const int so = m.slice_off[s.row / SLICE];
        nch = (m.slice_off[s.row / SLICE + 1] - so) / CHUNK_ROW;
        base = so + (s.row % SLICE) * 4;
        len = m.len[s.row]; j = m.order[s.row];
        if (s.part * CPS < nch) load_idx<CPS, I16>(c, m, base + s.part * CPS * CHUNK_ROW);
        lane_load(xj, tile_row(xprev + sub * V, j, pitch));
    }
    if (pdl) grid_dependency_wait();
    if (pdl == 2) grid_launch_dependents();
    float* vp = m.val + base;
    const float* dg = dk + sub * V;
    const int lim = len - ((G >= 4) ? sub / (G >= 4 ? G / 4 : 1) : (G == 2) ? 2 * sub : 0);
    // rows of a slice take the same number of steps; a group beyond its last one goes through the shuffles with the others
    const int most = __reduce_max_sync(0xffffffffu, nch);
    for (int t0 = 0; t0 < most; t0 += s.parts * CPS) {
        const int t = t0 + s.part * CPS;
        float4 w[CPS];
        Lane<V> d[4 * CPS];
        if (t < nch) {
#pragma unroll
            for (int i = 0; i < CPS; ++i) w[i] = __ldcs(reinterpret_cast<const float4*>(vp + (t + i) * CHUNK_ROW));
#pragma unroll
            for (int i = 0; i < CPS; ++i) { SDNN_GATHER_CHUNK(d, i, c[i], dg, pitch) }
            if (t + s.parts * CPS < nch) load_idx<CPS, I16>(c, m, base + (t + s.parts * CPS) * CHUNK_ROW);
        } else {
#pragma unroll
            for (int i = 0; i < CPS; ++i) {
                w[i] = make_float4(0.f, 0.f, 0.f, 0.f);
                lane_fill(d[4 * i], 0.f); lane_fill(d[4 * i + 1], 0.f); lane_fill(d[4 * i + 2], 0.f); lane_fill(d[4 * i + 3], 0.f);
            }
        }
        __syncwarp();
#pragma unroll
        for (int i = 0; i < CPS; ++i) {
            lane_fma(w[i].x, d[4 * i + 0], acc); lane_fma(w[i].y, d[4 * i + 1], acc);
            lane_fma(w[i].z, d[4 * i + 2], acc); lane_fma(w[i].w, d[4 * i + 3], acc);
            float p0 = lane_dot(d[4 * i + 0], xj), p1 = lane_dot(d[4 * i + 1], xj), p2 = lane_dot(d[4 * i + 2], xj), p3 = lane_dot(d[4 * i + 3], xj);
            chunk_sums<G>(p0, p1, p2, p3, sub, 0xffffffffu);
            chunk_update<G, false>(vp + (t + i) * CHUNK_ROW, nullptr, w[i], p0, p1, p2, p3, sub, (t + i) * 4, lim, step, inv_b);
        }
    }
    for (int o = G; o < G * s.parts; o <<= 1) lane_join(acc, o);
    if (s.row < n && s.part == 0) {
        lane_mask(acc, xj, act, clamp);
        lane_store(tile_row(dprev + sub * V, j, pitch), acc);
    }
    if (pdl == 1) grid_launch_dependents();
}

// ---------------------------------------------------------------------------------------------
// Layer kernels for tiles of padded width 4 (B <= 4: per-input SGD as in Algorithm 1, single vectors).
// With so few batch entries a row's work is its entries, not its batch: a lane per row (the mapping above) leaves a
// 1024-neuron layer to 32 warps that each walk 32 entries in four dependent steps.  Here a warp takes one SLICE of 16
// rows and a lane takes (row r = lane & 15, every second chunk starting at lane >> 4): the 32 lanes of one iteration
// read 512 contiguous bytes of indices and of values, up to EP_IT iterations (8 chunks, 32 entries per row) are in
// flight together, so a row of up to 32 entries costs one memory round trip for its entries and one for its
// gathers; the two lanes of a row add their partial sums with one shuffle.  Arithmetic per entry is the same as in
// the kernels above (lane_dot, fma(-step, g, w)), so the two copies of a layer stay bit-identical here too.
constexpr int EP_IT = 4;

struct EpShape { int lane, r, h, so, nch, item; };
__device__ __forceinline__ EpShape ep_shape(const Sliced& m, int n) {
    EpShape e;
    e.lane = threadIdx.x & 31; e.r = e.lane & 15; e.h = e.lane >> 4;
    const int s = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    const int ns = (n + SLICE - 1) / SLICE;
    e.so = 0; e.nch = 0; e.item = n;
    if (s < ns) {
        e.so = m.slice_off[s];
        e.nch = (m.slice_off[s + 1] - e.so) / CHUNK_ROW;
        e.item = min(n, s * SLICE + e.r);
    }
    return e;
}

#define SDNN_EP_LOAD_IDX(C, T0, IT)                                                                     \
    _Pragma("unroll") for (int i = 0; i < (IT); ++i) {                                                   \
        const int t = (T0) + 2 * i + e.h;                                                                \
        idx_zero(C[i]);                                                                                  \
        if (t < e.nch) load_idx4(C[i], m, e.so + t * CHUNK_ROW + e.r * 4);                               \
    }

template <bool I16>
__global__ void __launch_bounds__(128)
forward_ep_kernel(Sliced m, const float* __restrict__ bias, const float* __restrict__ xin, float* __restrict__ xout,
                  int n, float clamp, int act, int pdl) {
    const EpShape e = ep_shape(m, n);
    IdxChunk<I16> c[EP_IT];
    SDNN_EP_LOAD_IDX(c, 0, EP_IT)
    const float b = (e.item < n) ? bias[e.item] : 0.0f;
    const int to = (m.out && e.item < n) ? m.out[e.item] : e.item;
    if (pdl) grid_dependency_wait();
    if (pdl == 2) grid_launch_dependents();
    Lane<4> acc;
    lane_fill(acc, 0.0f);
    for (int t0 = 0; t0 < e.nch; t0 += 2 * EP_IT) {
        float4 w[EP_IT];
        Lane<4> x[4 * EP_IT];
#pragma unroll
        for (int i = 0; i < EP_IT; ++i) {
            const int t = t0 + 2 * i + e.h;
            w[i] = (t < e.nch) ? __ldcs(reinterpret_cast<const float4*>(m.val + e.so + t * CHUNK_ROW + e.r * 4)) : make_float4(0.f, 0.f, 0.f, 0.f);
        }
#pragma unroll
        for (int i = 0; i < EP_IT; ++i) { SDNN_GATHER_CHUNK(x, i, c[i], xin, 16u) }
        if (t0 + 2 * EP_IT < e.nch) { SDNN_EP_LOAD_IDX(c, t0 + 2 * EP_IT, EP_IT) }
#pragma unroll
        for (int i = 0; i < EP_IT; ++i) {
            lane_fma(w[i].x, x[4 * i + 0], acc); lane_fma(w[i].y, x[4 * i + 1], acc);
            lane_fma(w[i].z, x[4 * i + 2], acc); lane_fma(w[i].w, x[4 * i + 3], acc);
        }
    }
    acc.a.x += __shfl_xor_sync(0xffffffffu, acc.a.x, 16); acc.a.y += __shfl_xor_sync(0xffffffffu, acc.a.y, 16);
    acc.a.z += __shfl_xor_sync(0xffffffffu, acc.a.z, 16); acc.a.w += __shfl_xor_sync(0xffffffffu, acc.a.w, 16);
    if (e.h == 0 && e.item < n) {
        acc.a.x += b; acc.a.y += b; acc.a.z += b; acc.a.w += b;
        lane_activate(acc, act, clamp);
        lane_store(xout + (size_t)to * 4, acc);
    }
    if (pdl == 1) grid_launch_dependents();
}

// new values of the four entries of chunk t (positions 4t .. 4t+3 of a unit with `len` stored entries; padding keeps its 0)
__device__ __forceinline__ float4 ep_update(const float4& w, float p0, float p1, float p2, float p3, int t, int len, float step) {
    const int q = 4 * t;
    return make_float4(q + 0 < len ? __fmaf_rn(-step, p0, w.x) : w.x, q + 1 < len ? __fmaf_rn(-step, p1, w.y) : w.y,
                       q + 2 < len ? __fmaf_rn(-step, p2, w.z) : w.z, q + 3 < len ? __fmaf_rn(-step, p3, w.w) : w.w);
}

// Column units (transposed copy m): delta^{k-1}[j] = (sum_i w(i,j) delta^k[i]) (.) f'(x^{k-1}[j]) with the values before
// their update, and the update of the transposed copy's values.
// IT iterations (2 * IT chunks of a unit) in flight together.  The transposed copy's units are ragged (a column of a
// 32-per-row random pattern has 15 .. 55 entries): IT = 8 takes up to 64 entries in one go where the launch is bound by
// its chain of dependent round trips rather than by throughput (small nets).
template <int IT, bool I16>
__global__ void __launch_bounds__(128)
backward_col_ep_kernel(Sliced m, const float* __restrict__ xprev, const float* __restrict__ dk, float* __restrict__ dprev,
                       int n, float clamp, int act, const StepParams* __restrict__ sp, int pdl) {
    const EpShape e = ep_shape(m, n);
    IdxChunk<I16> c[IT];
    SDNN_EP_LOAD_IDX(c, 0, IT)
    int len = 0, j = 0;
    if (e.item < n) { len = m.len[e.item]; j = m.order[e.item]; }
    if (pdl) grid_dependency_wait();
    if (pdl == 2) grid_launch_dependents();
    const float step = sp->eta * sp->inv_b;
    Lane<4> xj, acc;
    lane_fill(xj, 0.0f); lane_fill(acc, 0.0f);
    if (e.item < n) lane_load(xj, xprev + (size_t)j * 4);
    for (int t0 = 0; t0 < e.nch; t0 += 2 * IT) {
        float4 w[IT];
        Lane<4> d[4 * IT];
#pragma unroll
        for (int i = 0; i < IT; ++i) {
            const int t = t0 + 2 * i + e.h;
            w[i] = (t < e.nch) ? ld_f4(m.val + e.so + t * CHUNK_ROW + e.r * 4) : make_float4(0.f, 0.f, 0.f, 0.f);
        }
#pragma unroll
        for (int i = 0; i < IT; ++i) { SDNN_GATHER_CHUNK(d, i, c[i], dk, 16u) }
        if (t0 + 2 * IT < e.nch) { SDNN_EP_LOAD_IDX(c, t0 + 2 * IT, IT) }
#pragma unroll
        for (int i = 0; i < IT; ++i) {
            const int t = t0 + 2 * i + e.h;
            lane_fma(w[i].x, d[4 * i + 0], acc); lane_fma(w[i].y, d[4 * i + 1], acc);
            lane_fma(w[i].z, d[4 * i + 2], acc); lane_fma(w[i].w, d[4 * i + 3], acc);
            if (t < e.nch)
                st_f4(m.val + e.so + t * CHUNK_ROW + e.r * 4,
                      ep_update(w[i], lane_dot(d[4 * i + 0], xj), lane_dot(d[4 * i + 1], xj), lane_dot(d[4 * i + 2], xj),
                                lane_dot(d[4 * i + 3], xj), t, len, step));
        }
    }
    acc.a.x += __shfl_xor_sync(0xffffffffu, acc.a.x, 16); acc.a.y += __shfl_xor_sync(0xffffffffu, acc.a.y, 16);
    acc.a.z += __shfl_xor_sync(0xffffffffu, acc.a.z, 16); acc.a.w += __shfl_xor_sync(0xffffffffu, acc.a.w, 16);
    if (e.h == 0 && e.item < n) {
        lane_mask(acc, xj, act, clamp);
        lane_store(dprev + (size_t)j * 4, acc);
    }
    if (pdl == 1) grid_launch_dependents();
}

// Row units (row-major copy m): update of its values (and of the bias) from delta^k[i] and the gathered x^{k-1}[j].
template <bool DBG, bool I16>
__global__ void __launch_bounds__(128)
backward_row_ep_kernel(Sliced m, float* __restrict__ bias, const float* __restrict__ xprev, const float* __restrict__ dk,
                       float* __restrict__ dbg_grad, int n, const StepParams* __restrict__ sp, int update_bias, int pdl) {
    const EpShape e = ep_shape(m, n);
    IdxChunk<I16> c[EP_IT];
    SDNN_EP_LOAD_IDX(c, 0, EP_IT)
    const int len = (e.item < n) ? m.len[e.item] : 0;
    const int lab = (m.out && e.item < n) ? m.out[e.item] : e.item;
    if (pdl) grid_dependency_wait();
    if (pdl == 2) grid_launch_dependents();
    const float inv_b = sp->inv_b;
    const float step = sp->eta * inv_b;
    Lane<4> d;
    lane_fill(d, 0.0f);
    if (e.item < n) lane_load(d, dk + (size_t)lab * 4);
    if (update_bias && e.h == 0 && e.item < n) bias[e.item] -= step * lane_sum(d);
    for (int t0 = 0; t0 < e.nch; t0 += 2 * EP_IT) {
        float4 w[EP_IT];
        Lane<4> x[4 * EP_IT];
#pragma unroll
        for (int i = 0; i < EP_IT; ++i) {
            const int t = t0 + 2 * i + e.h;
            w[i] = (t < e.nch) ? ld_f4(m.val + e.so + t * CHUNK_ROW + e.r * 4) : make_float4(0.f, 0.f, 0.f, 0.f);
        }
#pragma unroll
        for (int i = 0; i < EP_IT; ++i) { SDNN_GATHER_CHUNK(x, i, c[i], xprev, 16u) }
        if (t0 + 2 * EP_IT < e.nch) { SDNN_EP_LOAD_IDX(c, t0 + 2 * EP_IT, EP_IT) }
#pragma unroll
        for (int i = 0; i < EP_IT; ++i) {
            const int t = t0 + 2 * i + e.h;
            if (t < e.nch) {
                const float p0 = lane_dot(d, x[4 * i + 0]), p1 = lane_dot(d, x[4 * i + 1]), p2 = lane_dot(d, x[4 * i + 2]),
                            p3 = lane_dot(d, x[4 * i + 3]);
                const int at = e.so + t * CHUNK_ROW + e.r * 4;
                st_f4(m.val + at, ep_update(w[i], p0, p1, p2, p3, t, len, step));
                if (DBG) {
                    const int q = 4 * t;
                    st_f4(dbg_grad + at, make_float4(q + 0 < len ? p0 * inv_b : 0.f, q + 1 < len ? p1 * inv_b : 0.f,
                                                     q + 2 < len ? p2 * inv_b : 0.f, q + 3 < len ? p3 * inv_b : 0.f));
                }
            }
        }
    }
    if (pdl == 1) grid_launch_dependents();
}
#undef SDNN_EP_LOAD_IDX

// ---------------------------------------------------------------------------------------------
// Update of the row-major copy from the transposed one.  The column units have just computed the layer's new values, so the
// row-major copy only needs them moved: no second gather of x^{k-1} per entry, no second gradient, no old values.  Both copies
// are cut into blocks of `block` consecutive elements, and the move is two passes through shared memory with a buffer T between
// them, ordered by (block of the transposed copy, block of the row-major copy):
//   split_values : a CTA reads one block of the transposed copy and writes its part of T (both contiguous)
//   merge_values : a CTA collects its row-major block from the `nb` runs of T that belong to it (about 32 entries each: the
//                  block size is chosen for that) and writes it
// pos_a[t] / pos_b[t]: place of T's element t within its block of the transposed / row-major copy.  Nothing is scattered in
// global memory: fetching each value by its 4-byte address instead costs a request per entry (about one per clock and SM,
// 7 us for 2 M entries, and slower than the row units it would replace).  Per stored entry 20 bytes, all of it in order: split
// reads 4 + 2 (value, place) and writes 4, merge the same; the maps take 4 bytes an entry and the tables of runs some 0.4.  Alone
// on the device the two take 5.5 and 7.4 us for 0.5 M entries, two short launches of mostly round trips (143 CTAs of 256 threads at
// 32 and 64 registers, load pipe 5 and 12 % busy), which is why they run on four side streams beside the column units.
struct Move {
    const int* start;             // [nb * (nb + 1)] first element of run (block of the transposed copy, block of the row-major copy) in T
    const int2* runs;             // [nb * nb] the same by row-major block: (first element, length)
    const unsigned short* pos_a;
    const unsigned short* pos_b;
    int nb, block;
};
// Trained biases: b^k -= step * sum over the batch of delta^k (one more column of W^k whose input is the constant 1), a thread per
// stored row, in CTAs of the split launch behind those of the move: a launch of their own, which did not ask for the same split of an
// SM's memory, kept the column units waiting (6007 neurons, 37 inputs: 9.4 -> 7.8 us a layer).  n = 0: frozen.  The padding columns of delta are zero.
struct BiasUpdate { float* bias; const float* dk; const int* out; int n, ld; const StepParams* sp; };
constexpr int MOVE_THREADS = 256;
__global__ void __launch_bounds__(MOVE_THREADS, 4)
split_values_kernel(Move m, const float* __restrict__ cval, int c_elems, float* __restrict__ T, BiasUpdate u) {
    extern __shared__ __align__(16) float move_smem[];
    constexpr int AHEAD = 4;
    if ((int)blockIdx.x >= m.nb) {
        const int row = ((int)blockIdx.x - m.nb) * MOVE_THREADS + threadIdx.x;
        if (row >= u.n) return;
        const float* d = u.dk + (size_t)(u.out ? u.out[row] : row) * u.ld;
        float s = 0.0f;
        for (int b = 0; b < u.ld; b += 4) { const float4 v = ld_f4(d + b); s += (v.x + v.y) + (v.z + v.w); }
        u.bias[row] -= u.sp->eta * u.sp->inv_b * s;
        return;
    }
    const int cb = blockIdx.x, lo = cb * m.block, cnt = min(m.block, c_elems - lo);      // both multiples of 4
    for (int q = threadIdx.x * 4; q < cnt; q += MOVE_THREADS * 4) cp_async16(move_smem + q, cval + lo + q);
    cp_async_commit();
    const int t0 = m.start[cb * (m.nb + 1)], t1 = m.start[cb * (m.nb + 1) + m.nb];      // t0 a multiple of 4; T is padded to one
    ushort4 p[AHEAD];
    bool waited = false;
    for (int t = t0 + threadIdx.x * 4; __syncthreads_or(t < t1 || !waited); t += AHEAD * MOVE_THREADS * 4) {
#pragma unroll
        for (int i = 0; i < AHEAD; ++i)
            if (t + i * MOVE_THREADS * 4 < t1) p[i] = __ldcs(reinterpret_cast<const ushort4*>(m.pos_a + t + i * MOVE_THREADS * 4));
        if (!waited) { cp_async_wait<0>(); __syncthreads(); waited = true; }
#pragma unroll
        for (int i = 0; i < AHEAD; ++i)
            if (t + i * MOVE_THREADS * 4 < t1)
                st_f4(T + t + i * MOVE_THREADS * 4, make_float4(move_smem[p[i].x], move_smem[p[i].y], move_smem[p[i].z], move_smem[p[i].w]));
    }
}
__global__ void __launch_bounds__(MOVE_THREADS, 4)
merge_values_kernel(Move m, const float* __restrict__ T, float* __restrict__ rval, int r_elems) {
    extern __shared__ __align__(16) float move_smem[];
    constexpr int TEAMS = MOVE_THREADS / 16, RUNS = 4, DEEP = 3;                        // 16 threads share a run; 12 elements in flight per thread
    int2* runs = reinterpret_cast<int2*>(move_smem + m.block);
    const int rb = blockIdx.x, lo = rb * m.block, cnt = min(m.block, r_elems - lo);
    const int sub = threadIdx.x & 15, team = threadIdx.x >> 4;
    for (int q = threadIdx.x; q < m.nb; q += MOVE_THREADS) runs[q] = m.runs[(size_t)rb * m.nb + q];
    for (int q = threadIdx.x * 4; q < cnt; q += MOVE_THREADS * 4) st_f4(move_smem + q, make_float4(0.f, 0.f, 0.f, 0.f));      // padding
    __syncthreads();
    for (int cb = team; cb < m.nb; cb += TEAMS * RUNS) {
        int2 r[RUNS];
        float v[RUNS * DEEP];
        unsigned short at[RUNS * DEEP];
#pragma unroll
        for (int u = 0; u < RUNS; ++u) {
            r[u] = cb + u * TEAMS < m.nb ? runs[cb + u * TEAMS] : make_int2(0, 0);
#pragma unroll
            for (int d = 0; d < DEEP; ++d)
                if (sub + 16 * d < r[u].y) {
                    v[u * DEEP + d] = T[r[u].x + sub + 16 * d];
                    at[u * DEEP + d] = __ldcs(m.pos_b + r[u].x + sub + 16 * d);
                }
        }
#pragma unroll
        for (int u = 0; u < RUNS; ++u) {
#pragma unroll
            for (int d = 0; d < DEEP; ++d)
                if (sub + 16 * d < r[u].y) move_smem[at[u * DEEP + d]] = v[u * DEEP + d];
            for (int q = sub + 16 * DEEP; q < r[u].y; q += 16) move_smem[m.pos_b[r[u].x + q]] = T[r[u].x + q];
        }
    }
    __syncthreads();
    for (int q = threadIdx.x * 4; q < cnt; q += MOVE_THREADS * 4) __stcs(reinterpret_cast<float4*>(rval + lo + q), ld_f4(move_smem + q));
}
// Set-up of a Move, from `from` (place in the transposed copy of each element of the row-major copy, -1: padding): run lengths, the
// room of each block of the transposed copy in T (it begins at a multiple of 4), run starts, places.
__global__ void move_count_kernel(const int* __restrict__ from, int r_elems, int block, int nb, int* __restrict__ count) {
    for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < r_elems; e += gridDim.x * blockDim.x)
        if (from[e] >= 0) atomicAdd(count + (from[e] / block) * nb + e / block, 1);
}
constexpr int MOVE_SCAN = 256;
// sum over the CTA of v, in every thread; the CTA's threads all call it
__device__ __forceinline__ int move_sum(int v) {
    __shared__ int part[MOVE_SCAN / 32];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    __syncthreads();
    if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = v;
    __syncthreads();
    int sum = 0;
#pragma unroll
    for (int q = 0; q < MOVE_SCAN / 32; ++q) sum += part[q];
    return sum;
}
__global__ void __launch_bounds__(MOVE_SCAN) move_room_kernel(const int* __restrict__ count, int nb, int* __restrict__ room) {
    int c = 0;
    for (int rb = threadIdx.x; rb < nb; rb += MOVE_SCAN) c += count[blockIdx.x * nb + rb];
    c = move_sum(c);
    if (threadIdx.x == 0) room[blockIdx.x] = (c + 3) / 4 * 4;
}
// a CTA per block of the transposed copy; count: from here on the cursor of each run
__global__ void __launch_bounds__(MOVE_SCAN) move_starts_kernel(int* __restrict__ count, const int* __restrict__ room, int nb, int* __restrict__ start,
                                                                int2* __restrict__ runs) {
    __shared__ int warp_sum[MOVE_SCAN / 32];
    const int cb = blockIdx.x, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int at = 0;
    for (int q = threadIdx.x; q < cb; q += MOVE_SCAN) at += room[q];
    at = move_sum(at);
    for (int rb0 = 0; rb0 < nb; rb0 += MOVE_SCAN) {
        const int rb = rb0 + threadIdx.x, c = rb < nb ? count[cb * nb + rb] : 0;
        int upto = c;                                                                   // inclusive prefix within the warp
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) { const int v = __shfl_up_sync(0xffffffffu, upto, o); if (lane >= o) upto += v; }
        __syncthreads();
        if (lane == 31) warp_sum[warp] = upto;
        __syncthreads();
        int before = at, all = 0;
#pragma unroll
        for (int q = 0; q < MOVE_SCAN / 32; ++q) { before += q < warp ? warp_sum[q] : 0; all += warp_sum[q]; }
        if (rb < nb) {
            const int first = before + upto - c;
            start[cb * (nb + 1) + rb] = first; runs[(size_t)rb * nb + cb] = make_int2(first, c);
            count[cb * nb + rb] = first;
        }
        at += all;
    }
    if (threadIdx.x == 0) start[cb * (nb + 1) + nb] = at;
}
__global__ void move_places_kernel(const int* __restrict__ from, int r_elems, int block, int nb, int* __restrict__ cursor,
                                   unsigned short* __restrict__ pos_a, unsigned short* __restrict__ pos_b) {
    for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < r_elems; e += gridDim.x * blockDim.x) {
        const int p = from[e];
        if (p < 0) continue;
        const int t = atomicAdd(cursor + (p / block) * nb + e / block, 1);
        pos_a[t] = (unsigned short)(p % block); pos_b[t] = (unsigned short)(e % block);
    }
}

// ---------------------------------------------------------------------------------------------
// Fills the transposed copy's values from the row-major copy: entry (column j, row i) of the transposed
// copy is looked up by binary search in row i (ascending columns).  One warp per transposed unit.
// With `mismatch` non-NULL nothing is written; entries whose bits differ from the row-major copy are counted.
// row_of (or NULL): stored row of the row-major copy that holds neuron i, for layers whose rows are not in neuron order.
// from (or NULL): also notes where each entry of the row-major copy has its twin in the transposed one (see Move).
__global__ void mirror_values_kernel(Sliced rows, Sliced cols, int n, unsigned long long* mismatch, const int* __restrict__ row_of,
                                     int* __restrict__ from) {
    const int cc = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (cc >= n) return;
    const int len = cols.len[cc];
    const int j = cols.order[cc];
    const int base = cols.slice_off[cc / SLICE] + (cc % SLICE) * 4;
    for (int q = threadIdx.x & 31; q < len; q += 32) {
        const int pos = base + (q >> 2) * CHUNK_ROW + (q & 3);
        const int i = row_of ? row_of[load_idx1(cols, pos)] : load_idx1(cols, pos);
        const int rb = rows.slice_off[i / SLICE] + (i % SLICE) * 4;
        int lo = 0, hi = rows.len[i] - 1, at = -1;
        while (lo <= hi) {
            const int mid = (lo + hi) >> 1;
            const int c = load_idx1(rows, rb + (mid >> 2) * CHUNK_ROW + (mid & 3));
            if (c == j) { at = mid; break; }
            if (c < j) lo = mid + 1; else hi = mid - 1;
        }
        if (at < 0) { if (mismatch) atomicAdd(mismatch, 1ull << 32); continue; }     // pattern error: high word
        const float w = rows.val[rb + (at >> 2) * CHUNK_ROW + (at & 3)];
        if (from) from[rb + (at >> 2) * CHUNK_ROW + (at & 3)] = pos;
        if (mismatch) {
            if (__float_as_uint(w) != __float_as_uint(cols.val[pos])) atomicAdd(mismatch, 1ull);
        } else {
            cols.val[pos] = w;
        }
    }
}

// ---------------------------------------------------------------------------------------------
// The row-major copy's values in the caller's CSR order, and back (sdnn_get_weights / sdnn_set_weights).  Stored row s has
// its len[s] entries at start[s] .. of the caller's array (start NULL: at s * k, every row k long).  A warp takes a row: its
// side of the CSR array is contiguous, and the 16-byte pieces of the sliced side share their lines with the 15 other rows
// of the slice, which the warps of the same CTA read (both sides together run at HBM rate, 4 us for 2 M entries; what the
// calls wait for is the copy over PCIe).  TO_CSR false: CSR -> sliced.
template <bool TO_CSR>
__global__ void __launch_bounds__(512)
sliced_csr_kernel(Sliced m, float* __restrict__ csr, const int* __restrict__ start, int k, int n) {
    const int row = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (row >= n) return;
    const int len = m.len[row];
    const size_t at = start ? (size_t)start[row] : (size_t)row * k;
    float* v = m.val + m.slice_off[row / SLICE] + (row % SLICE) * 4;
    for (int q = threadIdx.x & 31; q < len; q += 32) {
        float& w = v[(q >> 2) * CHUNK_ROW + (q & 3)];
        if (TO_CSR) csr[at + q] = w; else w = csr[at + q];
    }
}

// ---------------------------------------------------------------------------------------------
// Dropping dead inputs during inference (inputs are independent of one another, Section 2; an input whose
// activation vector has become all zero stays all zero when no bias is positive).  The tile keeps its live
// inputs in its first *ncols columns; colmap[c] = position in the caller's tile of the input in column c.
//   cols_init : ncols = cnt, colmap = identity, flags cleared
//   live      : after a forward layer has marked the columns that still hold a nonzero: count them and - if that frees at least
//               one whole chunk of columns - renumber (perm[new] = old column, colmap follows, ncols = count, *do_compact = 1).
//               Single block; only after some of the layers, since renumbering costs two launches in the chain of layers
//   count     : live columns after every layer, from the marks, once per tile
//   compact   : moves the columns of every row to their new places, in place (a warp reads the part of a row it
//               is about to overwrite before it writes), and clears the rest of the last live chunk
//   expand    : final tile back to the caller's column positions, dead inputs all zero
struct ColState {
    int* ncols;        // live columns (device scalar)
    int* old_ncols;    // value of ncols before the last renumbering
    int* do_compact;
    int* colmap;       // [ld]
    int* perm;         // [ld]
    int* flags;        // [L][ld]: marks of each layer
};

__global__ void cols_init_kernel(ColState s, int cnt, int ld) {
    for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < ld; c += gridDim.x * blockDim.x) {
        s.colmap[c] = c; s.perm[c] = c;
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) { *s.ncols = cnt; *s.old_ncols = cnt; *s.do_compact = 0; }
}

__global__ void __launch_bounds__(1024) live_kernel(ColState s, const int* __restrict__ flags, int chunk) {
    __shared__ int warp_tot[32];
    __shared__ int carry, total;
    const int n = *s.ncols;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    // pass 1: how many columns are still live
    int cnt = 0;
    for (int b = threadIdx.x; b < n; b += 1024) cnt += (flags[b] != 0);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) cnt += __shfl_xor_sync(0xffffffffu, cnt, o);
    if (lane == 0) warp_tot[wid] = cnt;
    __syncthreads();
    if (threadIdx.x == 0) {
        int t = 0;
        for (int q = 0; q < 32; ++q) t += warp_tot[q];
        total = t; carry = 0;
    }
    __syncthreads();
    const int live = total;
    const bool renumber = (live + chunk - 1) / chunk < (n + chunk - 1) / chunk;
    if (renumber) {
        // pass 2: stable renumbering, 1024 columns at a time (new position <= old position)
        for (int base = 0; base < n; base += 1024) {
            const int b = base + threadIdx.x;
            const int f = (b < n && flags[b] != 0) ? 1 : 0;
            const int cm = (b < n) ? s.colmap[b] : 0;
            int incl = f;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int t = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= o) incl += t;
            }
            __syncthreads();                  // warp_tot free again; every colmap[b] of this round has been read
            if (lane == 31) warp_tot[wid] = incl;
            __syncthreads();
            int before = carry;
            for (int q = 0; q < wid; ++q) before += warp_tot[q];
            if (f) { const int np = before + incl - 1; s.perm[np] = b; s.colmap[np] = cm; }
            __syncthreads();
            if (threadIdx.x == 1023) carry = before + incl;
            __syncthreads();
        }
    }
    if (threadIdx.x == 0) {
        *s.do_compact = renumber ? 1 : 0;
        if (renumber) { *s.old_ncols = n; *s.ncols = live; }
    }
}

// a block per layer; columns that a layer did not process are not marked
__global__ void __launch_bounds__(256) live_count_kernel(const int* __restrict__ flags, int* __restrict__ live_after_layer, int ld) {
    __shared__ int part[8];
    int cnt = 0;
    for (int b = threadIdx.x; b < ld; b += 256) cnt += (flags[(size_t)blockIdx.x * ld + b] != 0);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) cnt += __shfl_xor_sync(0xffffffffu, cnt, o);
    if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = cnt;
    __syncthreads();
    if (threadIdx.x == 0) live_after_layer[blockIdx.x] = part[0] + part[1] + part[2] + part[3] + part[4] + part[5] + part[6] + part[7];
}

__global__ void __launch_bounds__(256) compact_kernel(ColState s, float* __restrict__ tile, int n, int ld, int chunk) {
    if (*s.do_compact == 0) return;
    const int live = *s.ncols;
    const int fill = min(ld, (live + chunk - 1) / chunk * chunk);       // columns the next layer will read
    const int lane = threadIdx.x & 31;
    const int warps = (gridDim.x * blockDim.x) >> 5;
    for (int row = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; row < n; row += warps) {
        float* r = tile + (size_t)row * ld;
        for (int base = 0; base < fill; base += 1024) {
            float v[32];
#pragma unroll
            for (int q = 0; q < 32; ++q) {
                const int c = base + q * 32 + lane;
                v[q] = (c < live) ? r[s.perm[c]] : 0.0f;
            }
            __syncwarp();
#pragma unroll
            for (int q = 0; q < 32; ++q) {
                const int c = base + q * 32 + lane;
                if (c < fill) r[c] = v[q];
            }
            __syncwarp();
        }
    }
}

__global__ void __launch_bounds__(256) expand_kernel(ColState s, const float* __restrict__ src, float* __restrict__ dst,
                                                     int n, int cols, int ld) {
    const int live = *s.ncols;
    const int lane = threadIdx.x & 31;
    const int warps = (gridDim.x * blockDim.x) >> 5;
    for (int row = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; row < n; row += warps) {
        const float* a = src + (size_t)row * ld;
        float* r = dst + (size_t)row * ld;
        for (int c = lane; c < cols; c += 32) r[c] = 0.0f;
        __syncwarp();
        for (int c = lane; c < live; c += 32) r[s.colmap[c]] = a[c];
    }
}

// ---------------------------------------------------------------------------------------------
// Probe of the bound of the layer kernels: nothing but random row gathers out of a table, with the indices made
// in registers (a linear congruential sequence per lane group, masked to the table), so that only the gathers
// use the load pipe.  G lanes of V floats per row (the layer kernels' own access width), eight gathers in flight
// per lane.
template <int G, int V, bool PAST_L1>
__global__ void __launch_bounds__(256)
gather_probe_kernel(const float* __restrict__ table, float* __restrict__ sink, unsigned row_mask, int per_group, unsigned seed) {
    const int tid = blockIdx.x * blockDim.x + threadIdx.x;
    const int sub = threadIdx.x % G;
    unsigned st = (unsigned)(tid / G) * 2654435761u + seed;
    float acc = 0.f;
    for (int q = 0; q < per_group; q += 8) {
        unsigned c[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) { st = st * 1664525u + 1013904223u; c[u] = (st >> 8) & row_mask; }
        Lane<V> v[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) lane_gather_sel<PAST_L1>(v[u], table + (size_t)c[u] * (V * G) + sub * V);
#pragma unroll
        for (int u = 0; u < 8; ++u) acc += lane_sum(v[u]);
    }
    if (acc == 123.456f) sink[0] = acc;      // the table is all zero: never taken, keeps the loads alive
}

// ---------------------------------------------------------------------------------------------
// How many rows must be in flight for the gather rate above?  The same 64-byte random rows (two lanes per row, one
// 256-bit load per lane), but in strict batches: a lane issues F loads, and the row numbers of its next batch depend on
// the sum of what these returned (always zero, which the compiler cannot know), so that exactly F loads per lane are
// in flight and nothing of the next batch starts before the last of them is back.  With T resident threads per SM that
// is T/2 * F rows in flight per SM; rows per clock against that number is the latency-throughput curve of the path, and
// rows in flight / rate is its round trip.
template <int F>
__global__ void __launch_bounds__(128, 1)
gather_inflight_probe_kernel(const float* __restrict__ table, float* __restrict__ sink, unsigned row_mask, int batches, unsigned seed) {
    const int tid = blockIdx.x * blockDim.x + threadIdx.x;
    const int sub = threadIdx.x & 1;
    unsigned st = (unsigned)(tid >> 1) * 2654435761u + seed;
    float acc = 0.f;
    for (int q = 0; q < batches; ++q) {
        unsigned c[F];
#pragma unroll
        for (int u = 0; u < F; ++u) { st = st * 1664525u + 1013904223u; c[u] = ((st >> 8) + __float_as_uint(acc)) & row_mask; }
        Lane<8> v[F];
#pragma unroll
        for (int u = 0; u < F; ++u) lane_gather(v[u], table + (size_t)c[u] * 16 + sub * 8);
#pragma unroll
        for (int u = 0; u < F; ++u) acc += lane_sum(v[u]);
    }
    if (acc == 123.456f) sink[0] = acc;      // the table is all zero: never taken, keeps the loads alive
}

// ---------------------------------------------------------------------------------------------
// What does a layer boundary cost?  Two ways to make every CTA's writes of one round visible to all CTAs of the next:
// a grid-wide barrier inside one cooperative launch (a release-add on a counter, then an acquire-spin until the
// round's count is reached: what a kernel that loops over the layers itself would pay per layer), and the end of one
// launch / start of the next under programmatic dependent launch (what the layer kernels pay).  Each round every thread
// writes one float, so that there is something to make visible.  The spin is bounded: a CTA that does not see its
// round complete within BARRIER_SPIN_LIMIT polls raises *err, and every CTA leaves at its next check.
constexpr int BARRIER_SPIN_LIMIT = 1 << 22;
__device__ __forceinline__ unsigned ld_acquire_gpu(const unsigned* p) {
    unsigned v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__global__ void grid_barrier_probe_kernel(unsigned* counter, int* err, int rounds, float* data) {
    const unsigned ctas = gridDim.x;
    for (int r = 0; r < rounds; ++r) {
        data[blockIdx.x * blockDim.x + threadIdx.x] = (float)r;
        __syncthreads();
        if (threadIdx.x == 0) {
            asm volatile("red.release.gpu.global.add.u32 [%0], %1;" :: "l"(counter), "r"(1u) : "memory");
            const unsigned want = (unsigned)(r + 1) * ctas;
            int spins = 0;
            while (ld_acquire_gpu(counter) < want)
                if (++spins > BARRIER_SPIN_LIMIT) { *err = 1; break; }
        }
        __syncthreads();
        if (*reinterpret_cast<volatile int*>(err)) return;
    }
}
__global__ void launch_chain_probe_kernel(float* data, int r) {
    grid_dependency_wait();
    grid_launch_dependents();
    data[blockIdx.x * blockDim.x + threadIdx.x] = (float)r;
}

// ---------------------------------------------------------------------------------------------
// Probe of the alternative to the second copy of the values: one value array in row-major order that the column
// units would read, or read and write, one 4-byte word at a time at scattered places (through a position map).  Eight
// accesses in flight per lane, indices made in registers.  STORE: 0 = scattered 4-byte loads, 1 = scattered 4-byte stores
// (every lane stores the value 0, so that the table stays all zero whatever the order).
template <int STORE>
__global__ void __launch_bounds__(256)
word_probe_kernel(float* __restrict__ table, float* __restrict__ sink, unsigned word_mask, int per_lane, unsigned seed) {
    const int tid = blockIdx.x * blockDim.x + threadIdx.x;
    unsigned st = (unsigned)tid * 2654435761u + seed;
    float acc = 0.f;
    for (int q = 0; q < per_lane; q += 8) {
        unsigned c[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) { st = st * 1664525u + 1013904223u; c[u] = (st >> 8) & word_mask; }
        if (STORE) {
#pragma unroll
            for (int u = 0; u < 8; ++u) table[c[u]] = 0.0f;
        } else {
            float v[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) v[u] = __ldg(table + c[u]);
#pragma unroll
            for (int u = 0; u < 8; ++u) acc += v[u];
        }
    }
    if (acc == 123.456f) sink[0] = acc;
}

// ---------------------------------------------------------------------------------------------
// The same probe for a table held in shared memory: of this CTA (cluster of 1), or spread over the shared memories of
// the CTAs of a thread-block cluster and read with ld.shared::cluster (distributed shared memory).  G lanes of 16 bytes
// per row (128-bit accesses: the widest shared-memory load), eight gathers in flight per lane.  Every CTA clears its
// part of the table; the cluster barriers before and after the gathers keep every CTA's shared memory alive while its
// neighbours read it.  rows_per_cta is a power of two; row r of the cluster's table lives in CTA r / rows_per_cta.
__device__ __forceinline__ void cluster_barrier() {
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ unsigned cluster_cta_rank() {
    unsigned r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}

template <int G, bool REMOTE>
__global__ void __launch_bounds__(1024)
smem_gather_probe_kernel(float* __restrict__ sink, unsigned rows_per_cta_log2, unsigned cluster_log2, int per_group, unsigned seed) {
    extern __shared__ __align__(16) float probe_table[];
    constexpr unsigned ROW_BYTES = 16u * G;
    const unsigned rows_per_cta = 1u << rows_per_cta_log2;
    for (unsigned q = threadIdx.x; q < rows_per_cta * (ROW_BYTES / 16u); q += blockDim.x)
        reinterpret_cast<float4*>(probe_table)[q] = make_float4(0.f, 0.f, 0.f, 0.f);
    __syncthreads();
    cluster_barrier();
    const unsigned base = (unsigned)__cvta_generic_to_shared(probe_table);
    const unsigned row_mask = (rows_per_cta << cluster_log2) - 1u;
    const int tid = blockIdx.x * blockDim.x + threadIdx.x;
    const unsigned sub = threadIdx.x % G;
    unsigned st = (unsigned)(tid / G) * 2654435761u + seed;
    float acc = 0.f;
    for (int q = 0; q < per_group; q += 8) {
        float4 v[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            st = st * 1664525u + 1013904223u;
            const unsigned r = (st >> 8) & row_mask;
            const unsigned addr = base + (r & (rows_per_cta - 1u)) * ROW_BYTES + sub * 16u;
            if (REMOTE) {
                unsigned ra;
                asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(ra) : "r"(addr), "r"(r >> rows_per_cta_log2));
                asm volatile("ld.shared::cluster.v4.f32 {%0,%1,%2,%3}, [%4];" : "=f"(v[u].x), "=f"(v[u].y), "=f"(v[u].z), "=f"(v[u].w) : "r"(ra));
            } else {
                asm volatile("ld.shared.v4.f32 {%0,%1,%2,%3}, [%4];" : "=f"(v[u].x), "=f"(v[u].y), "=f"(v[u].z), "=f"(v[u].w) : "r"(addr));
            }
        }
#pragma unroll
        for (int u = 0; u < 8; ++u) acc += (v[u].x + v[u].y) + (v[u].z + v[u].w);
    }
    if (acc == 123.456f) sink[0] = acc;      // the table is all zero: never taken, keeps the loads alive
    cluster_barrier();
}

// ---------------------------------------------------------------------------------------------
// The same probe for rows fetched by the copy engine (TMA) into shared memory instead of by load instructions into
// registers: GATHER4 = false: one cp.async.bulk of row_bytes per row; true: cp.async.bulk.tensor.2d ... tile::gather4,
// four rows of a two-dimensional tensor map (box: one row of row_bytes) per instruction.  The first `issuers` lanes of a
// warp issue one copy each per round into their own slot of a ring of TMA_STAGES stages per warp; a stage's copies complete on the warp's
// mbarrier for that stage.  Every wait on an mbarrier is bounded: after TMA_WAIT_LIMIT polls the warp records the
// failure in *status and stops issuing, waits (bounded again) for what it has in flight, and returns.
constexpr int TMA_STAGES = 4;
constexpr int TMA_WARPS = 4;
constexpr unsigned TMA_WAIT_LIMIT = 1u << 22;

__device__ __forceinline__ unsigned smem_u32(const void* p) { return (unsigned)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void mbar_init(unsigned bar, unsigned count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" :: "r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(unsigned bar, unsigned bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" :: "r"(bar), "r"(bytes) : "memory");
}
// polls until the phase with the given parity has completed; false if it gave up
__device__ __forceinline__ bool mbar_wait_bounded(unsigned bar, unsigned parity) {
    for (unsigned i = 0; i < TMA_WAIT_LIMIT; ++i) {
        unsigned done;
        asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
                     : "=r"(done) : "r"(bar), "r"(parity) : "memory");
        if (done) return true;
    }
    return false;
}

template <bool GATHER4>
__global__ void __launch_bounds__(32 * TMA_WARPS)
tma_gather_probe_kernel(const float* __restrict__ table, const __grid_constant__ CUtensorMap tmap, float* __restrict__ sink,
                        int* __restrict__ status, unsigned row_mask, unsigned row_bytes, int issuers, int rounds, unsigned seed) {
    extern __shared__ __align__(128) unsigned char tma_smem[];
    __shared__ __align__(8) unsigned long long bars[TMA_WARPS * TMA_STAGES];
    constexpr unsigned ROWS = GATHER4 ? 4u : 1u;                       // rows per copy
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const unsigned slot_bytes = ROWS * row_bytes;                      // one lane's copy
    const unsigned stage_bytes = (unsigned)issuers * slot_bytes;
    unsigned char* ring = tma_smem + (size_t)warp * TMA_STAGES * stage_bytes;
    if (lane == 0)
        for (int q = 0; q < TMA_STAGES; ++q) mbar_init(smem_u32(&bars[warp * TMA_STAGES + q]), 1u);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    __syncwarp();
    unsigned st = (unsigned)(blockIdx.x * blockDim.x + threadIdx.x) * 2654435761u + seed;
    float acc = 0.f;
    bool ok = true;
    int issued = 0;
    auto issue = [&](int r) {
        const int q = r % TMA_STAGES;
        const unsigned bar = smem_u32(&bars[warp * TMA_STAGES + q]);
        if (lane == 0) mbar_expect_tx(bar, stage_bytes);
        __syncwarp();
        const unsigned dst = smem_u32(ring + (size_t)q * stage_bytes + (size_t)lane * slot_bytes);
        if (lane >= issuers) return;
        if (GATHER4) {
            int r0, r1, r2, r3;
            st = st * 1664525u + 1013904223u; r0 = (int)((st >> 8) & row_mask);
            st = st * 1664525u + 1013904223u; r1 = (int)((st >> 8) & row_mask);
            st = st * 1664525u + 1013904223u; r2 = (int)((st >> 8) & row_mask);
            st = st * 1664525u + 1013904223u; r3 = (int)((st >> 8) & row_mask);
            asm volatile("cp.async.bulk.tensor.2d.shared::cluster.global.tile::gather4.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5, %6}], [%7];"
                         :: "r"(dst), "l"(reinterpret_cast<unsigned long long>(&tmap)), "r"(0), "r"(r0), "r"(r1), "r"(r2), "r"(r3), "r"(bar) : "memory");
        } else {
            st = st * 1664525u + 1013904223u;
            const unsigned long long src = reinterpret_cast<unsigned long long>(table) + (unsigned long long)((st >> 8) & row_mask) * row_bytes;
            asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                         :: "r"(dst), "l"(src), "r"(row_bytes), "r"(bar) : "memory");
        }
    };
    for (; issued < TMA_STAGES - 1 && issued < rounds; ++issued) issue(issued);
    int done = 0;
    for (; done < rounds && ok; ++done) {
        if (issued < rounds) {
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");      // the slot's earlier readers come before the engine's writes
            issue(issued); ++issued;
        }
        const int q = done % TMA_STAGES;
        ok = mbar_wait_bounded(smem_u32(&bars[warp * TMA_STAGES + q]), (unsigned)(done / TMA_STAGES) & 1u);
        ok = __all_sync(0xffffffffu, ok);
        if (ok && lane < issuers) acc += *reinterpret_cast<const float*>(ring + (size_t)q * stage_bytes + (size_t)lane * slot_bytes);
        __syncwarp();
    }
    if (!ok) {      // gave up: note it, then wait (bounded) for the copies still in flight before the shared memory goes away
        if (lane == 0) atomicExch(status, 1);
        for (; done < issued; ++done)
            mbar_wait_bounded(smem_u32(&bars[warp * TMA_STAGES + done % TMA_STAGES]), (unsigned)(done / TMA_STAGES) & 1u);
    }
    if (acc == 123.456f) sink[0] = acc;
}

// ---------------------------------------------------------------------------------------------
// Do the two gather paths add up?  One CTA of 1024 threads per SM: the first TMA_WARPS warps fetch rows with
// tile::gather4 into shared memory exactly as tma_gather_probe_kernel<true> does (tma_rounds rounds), the other 28 warps
// gather rows with 256-bit loads into registers exactly as gather_probe_kernel does (lsu_per_group rows per lane
// group), out of the same table.  Either part can be switched off by giving it no work.  If the paths are independent
// the launch takes as long as its slower part; if they share their bottleneck it takes the sum.
template <int G, int V>
__global__ void __launch_bounds__(1024)
mixed_gather_probe_kernel(const float* __restrict__ table, const __grid_constant__ CUtensorMap tmap, float* __restrict__ sink,
                          int* __restrict__ status, unsigned row_mask, int issuers, int tma_rounds, int lsu_per_group, unsigned seed) {
    extern __shared__ __align__(128) unsigned char tma_smem[];
    __shared__ __align__(8) unsigned long long bars[TMA_WARPS * TMA_STAGES];
    constexpr unsigned ROW_BYTES = 4u * G * V;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    unsigned st = (unsigned)(blockIdx.x * blockDim.x + threadIdx.x) * 2654435761u + seed;
    float acc = 0.f;
    if (warp >= TMA_WARPS) {      // ---- load path
        const int tid = blockIdx.x * (blockDim.x - 32 * TMA_WARPS) + (threadIdx.x - 32 * TMA_WARPS);
        const int sub = tid % G;
        st = (unsigned)(tid / G) * 2654435761u + seed;
        for (int q = 0; q < lsu_per_group; q += 8) {
            unsigned c[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) { st = st * 1664525u + 1013904223u; c[u] = (st >> 8) & row_mask; }
            Lane<V> v[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) lane_gather(v[u], table + (size_t)c[u] * (V * G) + sub * V);
#pragma unroll
            for (int u = 0; u < 8; ++u) acc += lane_sum(v[u]);
        }
        if (acc == 123.456f) sink[0] = acc;
        return;
    }
    // ---- copy-engine path (no CTA-wide barrier anywhere: the two kinds of warp never meet)
    const unsigned slot_bytes = 4u * ROW_BYTES, stage_bytes = (unsigned)issuers * slot_bytes;
    unsigned char* ring = tma_smem + (size_t)warp * TMA_STAGES * stage_bytes;
    if (lane == 0)
        for (int q = 0; q < TMA_STAGES; ++q) mbar_init(smem_u32(&bars[warp * TMA_STAGES + q]), 1u);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    __syncwarp();
    bool ok = true;
    int issued = 0;
    auto issue = [&](int r) {
        const int q = r % TMA_STAGES;
        const unsigned bar = smem_u32(&bars[warp * TMA_STAGES + q]);
        if (lane == 0) mbar_expect_tx(bar, stage_bytes);
        __syncwarp();
        if (lane >= issuers) return;
        const unsigned dst = smem_u32(ring + (size_t)q * stage_bytes + (size_t)lane * slot_bytes);
        int r0, r1, r2, r3;
        st = st * 1664525u + 1013904223u; r0 = (int)((st >> 8) & row_mask);
        st = st * 1664525u + 1013904223u; r1 = (int)((st >> 8) & row_mask);
        st = st * 1664525u + 1013904223u; r2 = (int)((st >> 8) & row_mask);
        st = st * 1664525u + 1013904223u; r3 = (int)((st >> 8) & row_mask);
        asm volatile("cp.async.bulk.tensor.2d.shared::cluster.global.tile::gather4.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5, %6}], [%7];"
                     :: "r"(dst), "l"(reinterpret_cast<unsigned long long>(&tmap)), "r"(0), "r"(r0), "r"(r1), "r"(r2), "r"(r3), "r"(bar) : "memory");
    };
    for (; issued < TMA_STAGES - 1 && issued < tma_rounds; ++issued) issue(issued);
    int done = 0;
    for (; done < tma_rounds && ok; ++done) {
        if (issued < tma_rounds) {
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            issue(issued); ++issued;
        }
        const int q = done % TMA_STAGES;
        ok = mbar_wait_bounded(smem_u32(&bars[warp * TMA_STAGES + q]), (unsigned)(done / TMA_STAGES) & 1u);
        ok = __all_sync(0xffffffffu, ok);
        if (ok && lane < issuers) acc += *reinterpret_cast<const float*>(ring + (size_t)q * stage_bytes + (size_t)lane * slot_bytes);
        __syncwarp();
    }
    if (!ok) {
        if (lane == 0) atomicExch(status, 1);
        for (; done < issued; ++done)
            mbar_wait_bounded(smem_u32(&bars[warp * TMA_STAGES + done % TMA_STAGES]), (unsigned)(done / TMA_STAGES) & 1u);
    }
    if (acc == 123.456f) sink[0] = acc;
}

// ---------------------------------------------------------------------------------------------
// Final-layer nonzero sets.  The tile is cut into segments of NZ_SEG rows and 32 columns, a block of 256 threads each.
//   count: bits[i/32][b] = which of 32 rows of column b are nonzero; seg_cnt[seg*ld + b] = how many of the segment's are
//   scan : per input b: nz_count[b] = total; seg_cnt becomes the exclusive prefix over segments
//   offs : exclusive scan of nz_count over the inputs of the tile, added to the running total
//   fill : ids written in ascending order at offs[b] + prefix[seg][b], a warp per column and segment, out of the bits
// (A thread per column and segment, its 256 rows one after the other, took 112 us to count 4096 x 1024 and 55 to fill.)
constexpr int NZ_SEG = 256;

__global__ void __launch_bounds__(256)
nz_count_kernel(const float* __restrict__ x, unsigned* __restrict__ bits, int* __restrict__ seg_cnt, int n, int cnt, int ld) {
    __shared__ int part[8][32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, b = blockIdx.y * 32 + lane;
    const int i0 = blockIdx.x * NZ_SEG + warp * 32;
    unsigned m = 0u;
    if (b < cnt) {
#pragma unroll 16
        for (int r = 0; r < 32; ++r)
            if (i0 + r < n) m |= (x[(size_t)(i0 + r) * ld + b] != 0.0f ? 1u : 0u) << r;
        if (i0 < n) bits[(size_t)(i0 >> 5) * ld + b] = m;
    }
    part[warp][lane] = __popc(m);
    __syncthreads();
    if (warp == 0 && b < cnt) {
        int c = 0;
#pragma unroll
        for (int q = 0; q < 8; ++q) c += part[q][lane];
        seg_cnt[(size_t)blockIdx.x * ld + b] = c;
    }
}

__global__ void nz_scan_segments_kernel(int* __restrict__ seg_cnt, int* __restrict__ tile_cnt, int nseg, int cnt, int ld) {
    const int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b >= cnt) return;
    int run = 0;
    for (int s0 = 0; s0 < nseg; s0 += 8) {
        int c[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) c[q] = s0 + q < nseg ? seg_cnt[(size_t)(s0 + q) * ld + b] : 0;
#pragma unroll
        for (int q = 0; q < 8; ++q)
            if (s0 + q < nseg) { seg_cnt[(size_t)(s0 + q) * ld + b] = run; run += c[q]; }
    }
    tile_cnt[b] = run;
}

// single block of 1024 threads: offs[b] = running + exclusive_scan(tile_cnt)[b]; running += total
__global__ void nz_scan_inputs_kernel(const int* __restrict__ tile_cnt, long long* __restrict__ offs,
                                      long long* __restrict__ running, int* __restrict__ count_out, int cnt) {
    __shared__ long long warp_tot[32];
    __shared__ long long carry;
    if (threadIdx.x == 0) carry = *running;
    __syncthreads();
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    for (int base = 0; base < cnt; base += 1024) {
        const int b = base + threadIdx.x;
        const long long v = (b < cnt) ? tile_cnt[b] : 0;
        long long incl = v;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            long long t = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += t;
        }
        if (lane == 31) warp_tot[wid] = incl;
        __syncthreads();
        if (wid == 0) {
            long long w = warp_tot[lane], wi = w;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                long long t = __shfl_up_sync(0xffffffffu, wi, o);
                if (lane >= o) wi += t;
            }
            warp_tot[lane] = wi - w;   // exclusive prefix of the warp totals
        }
        __syncthreads();
        const long long excl = carry + warp_tot[wid] + incl - v;
        if (b < cnt) {
            offs[b] = excl;
            if (count_out) count_out[b] = (int)v;
        }
        __syncthreads();
        if (threadIdx.x == 1023) carry = excl + v;
        __syncthreads();
    }
    if (threadIdx.x == 0) *running = carry;
}

__global__ void __launch_bounds__(256)
nz_fill_kernel(const unsigned* __restrict__ bits, const int* __restrict__ seg_pre, const long long* __restrict__ offs, int* __restrict__ out,
               long long capacity, int n, int cnt, int ld) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int i = blockIdx.x * NZ_SEG + lane * 8;                       // a lane takes eight rows of the segment
    for (int q = 0; q < 4; ++q) {
        const int b = blockIdx.y * 32 + warp * 4 + q;
        if (b >= cnt) return;
        unsigned m = i < n ? (bits[(size_t)(i >> 5) * ld + b] >> (i & 31)) & 0xffu : 0u;
        int before = __popc(m);
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int v = __shfl_up_sync(0xffffffffu, before, o);
            if (lane >= o) before += v;
        }
        long long pos = offs[b] + seg_pre[(size_t)blockIdx.x * ld + b] + before - __popc(m);
        while (m) {
            if (pos < capacity) out[pos] = i + __ffs(m) - 1;
            ++pos;
            m &= m - 1;
        }
    }
}

}  // namespace sdnn_kernels
