// A whole network for one to four inputs in one launch (per-input latency, narrow nets).
//
// A layer of 1024 neurons and one input is 32 K multiply-adds: as a launch of its own it takes 1.7 us, all of it launch,
// prologue and round trips, and a chain of 120 launches costs the host as much again.  Here a cluster of 16 CTAs runs all layers:
// each CTA has all activations in its shared memory and computes a sixteenth of the rows, four lanes per row; the partial sums
// meet in shuffles, the CTA's outputs are collected in its shared memory and copied to every CTA of the cluster in one bulk copy
// each, which counts its bytes down on the receiver's mbarrier.  A CTA goes on to the next layer when all n values have
// arrived: no cluster-wide barrier in the chain.  Two buffers are enough: a CTA sends layer k + 1 after it has received all of layer
// k, and a CTA sends its part of layer k after its last read of layer k - 1.  What bounds a layer is that chain: read, add,
// collect, send, arrive.  The argument needs every CTA that is sent to to send as well: a CTA that sent nothing would be waited for by
// nobody, and the others could be two layers ahead of it, counting on a barrier whose last phase it has not seen the end of.  A
// net of at most 960 neurons leaves CTAs without rows: they take no part in the exchange (vector_ctas).
// The entries are off the chain: a CTA's part of a layer is one contiguous stretch of the sliced copy, and
// bulk copies bring it into a ring of shared-memory stages several layers ahead.  (Prefetched into registers two layers ahead
// instead, a layer takes 1.0 us as well: either way the entries are not what it waits for, and the ring needs no registers for them.)
// The launch: 16 CTAs of 256 threads, 80 registers; under ncu 132 us for 120 layers of 1024, the issue slots of its 16 SMs 27 % busy,
// shared-memory wavefronts 20 % of what those SMs could do, 43 % of them bank conflicts of the random reads: latency, not a pipe.
// Every wait is bounded: after VECTOR_WAIT_LIMIT polls the thread raises *status, waits no more and ends with the others.  From then
// on it sends nothing, loads nothing and arms no barrier: a barrier whose phase it has not seen the end of must not be counted
// on again, and every copy it has issued is older than the wait that it gave up.  CTAs that miss what it would have sent give up
// in their turn.  Nor does it gather: indices that have not arrived could point anywhere.  No CTA leaves the cluster before the last.
#pragma once
#include "kernels.cuh"
#include "plan.h"

namespace sdnn_kernels {

using namespace sdnn_plan;
constexpr int VECTOR_THREADS = 256, VECTOR_WARPS = VECTOR_THREADS / 32;
static_assert(VECTOR_BLOCK == VECTOR_WARPS * 8 && VECTOR_CTAS == 2 * VECTOR_WARPS, "eight rows a warp; a warp sends to two CTAs");
constexpr int VECTOR_STAGES = 8;                             // most stages of the ring of entries
constexpr unsigned VECTOR_WAIT_LIMIT = 1u << 20;

struct VectorLayer {
    const unsigned short* idx;      // row-major sliced copy, 16-bit indices
    const float* val;
};
struct VectorArgs {
    const VectorLayer* layers;      // [depth]
    const float* bias;              // [depth][n]
    int n, depth;
    int ctas;                       // CTAs that have rows (vector_ctas): the others only hold their place in the cluster
    int kpad;                       // entries per row of every slice of every layer (a multiple of 8)
    int stages;                     // of the ring of entries
    const float* x;                 // [cnt][n]
    int cnt;
    float* y;                       // [cnt][n] or NULL
    int* nz_count;                  // [cnt] or NULL
    float* acts;                    // training: tiles [depth + 1][n][4] of x^0 (read instead of x) and x^1 .. (written); else NULL
    int* status;
    float clamp;
    int act;
};

template <int V> struct Vec { float a[V]; };
__device__ __forceinline__ void vec_ld(Vec<1>& v, unsigned p) { asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v.a[0]) : "r"(p)); }
__device__ __forceinline__ void vec_ld(Vec<2>& v, unsigned p) { asm volatile("ld.shared.v2.f32 {%0, %1}, [%2];" : "=f"(v.a[0]), "=f"(v.a[1]) : "r"(p)); }
__device__ __forceinline__ void vec_ld(Vec<4>& v, unsigned p) {
    asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.a[0]), "=f"(v.a[1]), "=f"(v.a[2]), "=f"(v.a[3]) : "r"(p));
}
__device__ __forceinline__ void vec_st(unsigned p, const Vec<1>& v) { asm volatile("st.shared.f32 [%0], %1;" :: "r"(p), "f"(v.a[0]) : "memory"); }
__device__ __forceinline__ void vec_st(unsigned p, const Vec<2>& v) { asm volatile("st.shared.v2.f32 [%0], {%1, %2};" :: "r"(p), "f"(v.a[0]), "f"(v.a[1]) : "memory"); }
__device__ __forceinline__ void vec_st(unsigned p, const Vec<4>& v) {
    asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};" :: "r"(p), "f"(v.a[0]), "f"(v.a[1]), "f"(v.a[2]), "f"(v.a[3]) : "memory");
}
// address of the same shared-memory location in another CTA of the cluster
__device__ __forceinline__ unsigned cluster_addr(unsigned p, unsigned rank) {
    unsigned r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(p), "r"(rank));
    return r;
}
// bytes (a multiple of 16) of this CTA's shared memory to another one's, counted down on the barrier there; dst and bar:
// shared::cluster addresses in the same CTA
__device__ __forceinline__ void send_bulk(unsigned dst, unsigned src, unsigned bytes, unsigned bar) {
    asm volatile("cp.async.bulk.shared::cluster.shared::cta.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 :: "r"(dst), "r"(src), "r"(bytes), "r"(bar) : "memory");
}
__device__ __forceinline__ void load_bulk(unsigned dst, const void* src, unsigned bytes, unsigned bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 :: "r"(dst), "l"(src), "r"(bytes), "r"(bar) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait_cluster(unsigned bar, unsigned parity) {
    unsigned done;
    asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
                 : "=r"(done) : "r"(bar), "r"(parity) : "memory");
    return done != 0u;
}
// waits for the phase of the given parity; false once *status has been raised by this thread
__device__ __forceinline__ bool vector_wait(bool ok, unsigned bar, unsigned parity, int* status) {
    if (!ok) return false;
    unsigned polls = 0;
    while (!mbar_try_wait_cluster(bar, parity)) if (++polls > VECTOR_WAIT_LIMIT) { *status = 1; return false; }
    return true;
}

template <int V>
__global__ void __launch_bounds__(VECTOR_THREADS, 1)
vector_infer_kernel(const VectorArgs a) {
    // two activation buffers [n][V], two send buffers [rows of the CTA][V], the layers' table, the ring: per stage the values and the
    // indices of the CTA's blocks, in the sliced layout
    extern __shared__ __align__(128) unsigned char vector_smem[];
    __shared__ __align__(8) unsigned long long bars[2 + VECTOR_STAGES];
    __shared__ int counts[4];
    constexpr unsigned PITCH = V * 4u;
    constexpr int STRIDE = VECTOR_CTAS * VECTOR_BLOCK;                                    // rows between two blocks of a CTA
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int e = lane >> 3;                                                              // a lane takes chunks e, e + 4, ... of its row
    const unsigned rank = cluster_cta_rank();
    const int n = a.n, per_layer = (n + STRIDE - 1) / STRIDE, nch = a.kpad / 4;
    const unsigned x0 = smem_u32(vector_smem), x_bytes = ((unsigned)n * PITCH + 15u) & ~15u;
    const unsigned s0 = x0 + 2 * x_bytes, s_bytes = (unsigned)per_layer * VECTOR_BLOCK * PITCH, bar0 = smem_u32(&bars[0]);
    const unsigned block_elems = (unsigned)(VECTOR_BLOCK * a.kpad), val_bytes = (unsigned)per_layer * block_elems * 4u, stage_bytes = val_bytes / 2 * 3;
    VectorLayer* table = reinterpret_cast<VectorLayer*>(vector_smem + 2 * x_bytes + 2 * s_bytes);
    const unsigned ring = (s0 + 2 * s_bytes + (unsigned)(a.depth * sizeof(VectorLayer)) + 127u) & ~127u;
    if (threadIdx.x == 0)
        for (int q = 0; q < 2 + VECTOR_STAGES; ++q) mbar_init(bar0 + q * 8u, 1u);
    if (threadIdx.x < 4) counts[threadIdx.x] = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    for (int q = threadIdx.x; q < a.depth; q += VECTOR_THREADS) table[q] = a.layers[q];
    // the input vectors, in every CTA
    for (int i = threadIdx.x; i < n; i += VECTOR_THREADS)
#pragma unroll
        for (int b = 0; b < V; ++b)
            reinterpret_cast<float*>(vector_smem)[i * V + b] = a.acts ? a.acts[i * 4 + b] : b < a.cnt ? a.x[(size_t)b * n + i] : 0.0f;
    const unsigned ctas = (unsigned)a.ctas;
    // receivers: warp w sends to CTAs w and w + 8, those of them that have rows
    const unsigned my_x = x0 + rank * (VECTOR_BLOCK * PITCH);
    const unsigned to_x[2] = {cluster_addr(my_x, warp), cluster_addr(my_x, warp + VECTOR_WARPS)};
    const unsigned to_bar[2] = {cluster_addr(bar0, warp), cluster_addr(bar0, warp + VECTOR_WARPS)};
    __syncthreads();

    // entries of layer k into its stage (one thread)
    auto load = [&](int k) {
        const int stage = k % a.stages;
        const unsigned bar = bar0 + (2 + stage) * 8u, val = ring + stage * stage_bytes, idx = val + val_bytes;
        unsigned total = 0;
        for (int d = 0; d < per_layer; ++d) {
            const int row = (int)rank * VECTOR_BLOCK + d * STRIDE, rows = min(VECTOR_BLOCK, (n + SLICE - 1) / SLICE * SLICE - row);
            if (rows > 0) total += (unsigned)(rows * a.kpad) * 6u;
        }
        mbar_expect_tx(bar, total);
        for (int d = 0; d < per_layer; ++d) {
            const int row = (int)rank * VECTOR_BLOCK + d * STRIDE, rows = min(VECTOR_BLOCK, (n + SLICE - 1) / SLICE * SLICE - row);
            if (rows > 0) {
                const unsigned elems = (unsigned)(rows * a.kpad);
                load_bulk(val + d * block_elems * 4u, table[k].val + (size_t)row * a.kpad, elems * 4u, bar);
                load_bulk(idx + d * block_elems * 2u, table[k].idx + (size_t)row * a.kpad, elems * 2u, bar);
            }
        }
    };
    if (threadIdx.x == 0 && rank < ctas)
        for (int k = 0; k < min(a.stages, a.depth); ++k) load(k);

    const int row0 = (int)rank * VECTOR_BLOCK + warp * 8 + (lane & 7);                    // this lane's row in block 0
    // its first chunk in a block: slice (warp / 2) of the block, row (warp % 2) * 8 + lane % 8 of the slice
    const unsigned in_block = (unsigned)((warp >> 1) * SLICE * a.kpad + ((warp & 1) * 8 + (lane & 7)) * 4 + e * CHUNK_ROW);
    float bias[4];                                                                        // of the next layer's first four blocks
    auto next_bias = [&](int k) {
#pragma unroll
        for (int d = 0; d < 4; ++d) if (d < per_layer) bias[d] = a.bias[(size_t)min(k, a.depth - 1) * n + min(row0 + d * STRIDE, n - 1)];
    };
    next_bias(0);
    cluster_barrier();
    if (rank >= ctas) { cluster_barrier(); return; }                                      // no rows: nobody sends to it, it waits for nothing
    if (threadIdx.x == 0) mbar_expect_tx(bar0 + 8u, x_bytes);

    bool ok = true;
    int stage = 0;
    unsigned stage_phase = 0u;
    // layer k reads buffer k % 2; its outputs arrive in the other one and are counted on that one's barrier
    unsigned in = x0, send = s0, out_off = x_bytes, bar_off = 8u, phase = 0u;
    for (int k = 0; k < a.depth; ++k) {
        ok = vector_wait(ok, bar0 + (2 + stage) * 8u, stage_phase, a.status);             // the layer's entries: long there
        const unsigned val = ring + stage * stage_bytes + in_block * 4u, idx = ring + stage * stage_bytes + val_bytes + in_block * 2u;
#pragma unroll 1
        for (int d = 0; d < per_layer; ++d) {
            Vec<V> acc0, acc1;
#pragma unroll
            for (int b = 0; b < V; ++b) { acc0.a[b] = 0.0f; acc1.a[b] = 0.0f; }
            auto chunk = [&](Vec<V>& acc, int t) {
                unsigned ca, cb;
                asm volatile("ld.shared.v2.u32 {%0, %1}, [%2];" : "=r"(ca), "=r"(cb) : "r"(idx + (d * block_elems + t * CHUNK_ROW) * 2u));
                Vec<4> w;
                vec_ld(w, val + (d * block_elems + t * CHUNK_ROW) * 4u);
                Vec<V> g0, g1, g2, g3;
                vec_ld(g0, in + (ca & 0xffffu) * PITCH); vec_ld(g1, in + (ca >> 16) * PITCH);
                vec_ld(g2, in + (cb & 0xffffu) * PITCH); vec_ld(g3, in + (cb >> 16) * PITCH);
#pragma unroll
                for (int b = 0; b < V; ++b)
                    acc.a[b] = fmaf(w.a[3], g3.a[b], fmaf(w.a[2], g2.a[b], fmaf(w.a[1], g1.a[b], fmaf(w.a[0], g0.a[b], acc.a[b]))));
            };
            const int mine = ok && row0 + d * STRIDE < n ? nch : 0;                       // the stage holds nothing for rows beyond the last one
            int t = 0;
            for (; t + 4 + e < mine; t += 8) { chunk(acc0, t); chunk(acc1, t + 4); }
            if (t + e < mine) chunk(acc0, t);
#pragma unroll
            for (int b = 0; b < V; ++b) acc0.a[b] += acc1.a[b];
#pragma unroll
            for (int o = 8; o < 32; o <<= 1)
#pragma unroll
                for (int b = 0; b < V; ++b) acc0.a[b] += __shfl_xor_sync(0xffffffffu, acc0.a[b], o);
            if (e == 0) {
                const float bb = d == 0 ? bias[0] : d == 1 ? bias[1] : d == 2 ? bias[2] : bias[3];
#pragma unroll
                for (int b = 0; b < V; ++b) acc0.a[b] = a.act == ACT_SIGMOID ? activate(acc0.a[b] + bb, ACT_SIGMOID, a.clamp) : clampf(acc0.a[b] + bb, a.clamp);
                vec_st(send + (unsigned)(d * VECTOR_BLOCK + warp * 8 + lane) * PITCH, acc0);
                if (a.acts && row0 + d * STRIDE < n) {
                    float4 v = make_float4(acc0.a[0], 0.f, 0.f, 0.f);
                    if (V > 1) v.y = acc0.a[V > 1 ? 1 : 0];
                    if (V > 2) { v.z = acc0.a[V > 2 ? 2 : 0]; v.w = acc0.a[V > 2 ? 3 : 0]; }
                    st_f4(a.acts + ((size_t)(k + 1) * n + row0 + d * STRIDE) * 4, v);
                }
            }
        }
        __syncthreads();
        if (lane == 0 && ok) {
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            for (int s = 0; s < per_layer; ++s) {
                const int rows = min(VECTOR_BLOCK, n - ((int)rank * VECTOR_BLOCK + s * STRIDE));
                if (rows <= 0) break;
                const unsigned bytes = ((unsigned)rows * PITCH + 15u) & ~15u, off = out_off + (unsigned)(s * STRIDE) * PITCH;
                if (warp < ctas) send_bulk(to_x[0] + off, send + (unsigned)(s * VECTOR_BLOCK) * PITCH, bytes, to_bar[0] + bar_off);
                if (warp + VECTOR_WARPS < ctas) send_bulk(to_x[1] + off, send + (unsigned)(s * VECTOR_BLOCK) * PITCH, bytes, to_bar[1] + bar_off);
            }
            if (warp == 0 && k + a.stages < a.depth) load(k + a.stages);                  // every warp has read this layer's stage
        }
        __syncwarp();
        next_bias(k + 1);
        ok = vector_wait(ok, bar0 + bar_off, phase, a.status);
        in = x0 + out_off;
        if (++stage == a.stages) { stage = 0; stage_phase ^= 1u; }
        if (bar_off == 8u) { bar_off = 0u; out_off = 0u; send += s_bytes; }
        else { bar_off = 8u; out_off = x_bytes; send -= s_bytes; phase ^= 1u; }           // both barriers have completed once more
        // this barrier's last phase is over: it counts the next layer
        if (threadIdx.x == 0 && ok && k + 1 < a.depth) mbar_expect_tx(bar0 + bar_off, x_bytes);
    }

    const float* x = reinterpret_cast<const float*>(vector_smem + ((a.depth & 1) ? x_bytes : 0u));
    if (a.y)
        for (int i = (int)rank * VECTOR_THREADS + threadIdx.x; i < n; i += a.ctas * VECTOR_THREADS)
#pragma unroll
            for (int b = 0; b < V; ++b) if (b < a.cnt) a.y[(size_t)b * n + i] = x[i * V + b];
    if (a.nz_count && rank == 0) {
        __syncthreads();
#pragma unroll
        for (int b = 0; b < V; ++b) {
            int c = 0;
            for (int i = threadIdx.x; i < n; i += VECTOR_THREADS) c += x[i * V + b] != 0.0f;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) c += __shfl_xor_sync(0xffffffffu, c, o);
            if (lane == 0 && c) atomicAdd(counts + b, c);
        }
        __syncthreads();
        if (threadIdx.x < a.cnt) a.nz_count[threadIdx.x] = counts[threadIdx.x];
    }
    cluster_barrier();      // no CTA leaves while another may still write to its shared memory
}

}  // namespace sdnn_kernels
