// Segments of small steps in one launch (sm_103a).
//
// A circuit network is full of steps on gate-sized tensors: products of 4 to 4096 entries that take
// well under a microsecond each, against 3 to 5 us for a launch of their own, and against about 5 us
// a step for a CTA that reads every operand and descriptor from global memory in plan order.  k_seg
// runs a whole connected group of them: the program and every intermediate sit in shared memory, the
// steps are grouped into stages by their depth in the contraction tree, and a stage's steps are
// spread over the CTA's warps in pieces of 32 outputs, so a stage costs one block barrier and
// a few hundred clocks.  What bounds it for few items is that latency times the depth, not bytes or
// flops; for thousands of items it is shared-memory bank conflicts of the strided operand reads, and
// the compiler's rule (seg_pays, qx_host.cpp) leaves those to launches per step.
// Measured: the 265 invariant steps of the 20-qubit sliced plan 224 -> 16 us (41 segments, one launch);
// a 12-qubit call of 17 bitstrings 208 -> 67 us (31 -> 5 launches); one amplitude of 16 qubits, depth
// 12: 780 -> 212 us (287 -> 21 launches); the 36-qubit local-search plan 774 -> 77 launches.
//
// Every output is the sum over k in increasing order with the same FMA sequence, folded every 64 k,
// as in the one-launch-per-step kernels, so both give the same bits.
#include <mutex>

#include "qx_seg.h"

namespace qx {

namespace {

__device__ __forceinline__ void seg_fma(float2& acc, float2 a, float2 b) {
    acc.x = fmaf(a.x, b.x, acc.x);
    acc.x = fmaf(-a.y, b.y, acc.x);
    acc.y = fmaf(a.x, b.y, acc.y);
    acc.y = fmaf(a.y, b.x, acc.y);
}

// sum of t[b] over the set bits b of v
__device__ __forceinline__ uint32_t strides(uint32_t v, const uint32_t* t) {
    uint32_t s = 0;
    for (int b = 0; v >> b; ++b)
        if ((v >> b) & 1) s += t[b];
    return s;
}
// ... over the five bits of a lane number (t 16-byte aligned, one step: no loop, two vector loads)
__device__ __forceinline__ uint32_t lane_strides(int lane, const uint32_t* t) {
    const uint4 a = *(const uint4*)t;
    const uint32_t e = t[4];
    return ((lane & 1) ? a.x : 0u) + ((lane & 2) ? a.y : 0u) + ((lane & 4) ? a.z : 0u) + ((lane & 8) ? a.w : 0u) +
           ((lane & 16) ? e : 0u);
}

__device__ __forceinline__ int64_t in_offset(const SegIn& in, const SegCtx& c, int64_t item) {
    const uint32_t nb = (uint32_t)c.ic.n_b, sl = (uint32_t)item / nb;
    int64_t off = in.off;
    if (in.space == SEG_SLICE) off = off * c.cap[1] + ((int64_t)(c.per_pair ? sl : (uint32_t)item) << in.rank);
    else if (in.space == SEG_PAIR) off = off * c.cap[2] + (item << in.rank);
    if (in.n_fix) {
        const int64_t s = c.ic.s0 + sl, b = c.ic.b0 + ((uint32_t)item - sl * nb);
        for (int f = 0; f < in.n_fix; ++f) {
            const int src = in.fix_src[f];
            const int64_t v = src >= 0 ? (s >> src) & 1 : (int64_t)(c.ic.bits[b * c.ic.n_qubits - src - 1] & 1);
            off += v * in.fix_stride[f];
        }
    }
    return off;
}

// copies the operands of `item` into the arena (once: only those that every item shares): 16 threads
// per tiny operand (several of them in flight per thread), the whole CTA for each larger one
__device__ __forceinline__ void load_one(const SegIn& in, const SegCtx& c, int64_t item, int e, int step, float2* arena) {
    const float2* src = (in.space == SEG_LEAF ? c.leaves : c.region[in.space]) + in_offset(in, c, item);
    const int n = 1 << in.rank;
#pragma unroll 4
    for (; e < n; e += step) {
        int64_t a = e;
        if (!in.natural) {
            a = 0;
            for (int b = 0; b < in.rank; ++b)
                if ((e >> b) & 1) a += (int64_t)1 << in.pos[b];
        }
        arena[in.arena + e] = src[a];
    }
}
__device__ __forceinline__ void load_inputs(const SegIn* ins, int n_tiny, int n_in, const SegCtx& c, int64_t item,
                                            bool once, float2* arena) {
    const int groups = blockDim.x >> 4, e = threadIdx.x & 15;
#pragma unroll 4
    for (int i = threadIdx.x >> 4; i < n_tiny; i += groups)
        if ((ins[i].once != 0) == once) load_one(ins[i], c, item, e, 16, arena);
    for (int i = n_tiny; i < n_in; ++i)
        if ((ins[i].once != 0) == once) load_one(ins[i], c, item, threadIdx.x, blockDim.x, arena);
}

// acc += X[a_k] Y[a_k] for k = k0 .. k0 + N - 1, loads ahead of the sums
template <int N>
__device__ __forceinline__ void mac(float2& acc, const float2* X, const float2* Y, uint32_t base, uint32_t klane, int k0) {
    float2 x[N], y[N];
#pragma unroll
    for (int j = 0; j < N; ++j) {
        const uint32_t a = base + __shfl_sync(0xffffffffu, klane, k0 + j);
        x[j] = X[a & 0xffff];
        y[j] = Y[a >> 16];
    }
#pragma unroll
    for (int j = 0; j < N; ++j) seg_fma(acc, x[j], y[j]);
}

__device__ __forceinline__ void run_task(const SegOp& op, const SegTask& t, float2* arena, float2* result) {
    const int lane = threadIdx.x & 31;
    const float2* X = arena + op.x;
    const float2* Y = arena + op.y;
    float2* D = (op.dst < 0 ? result : arena + op.dst) + t.d;
    const int kb = op.kb;
    if (op.kind == SEGOP_DOT) {
        // 256 partials over k = p, p + 256, ..., lane holding p = lane + 32 j, then a halving tree
        const int K = 1 << kb;
        float2 r[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            r[j] = make_float2(0.f, 0.f);
            for (int k = lane + 32 * j; k < K; k += 256) {
                const uint32_t a = t.xy + strides(k, op.k);
                seg_fma(r[j], X[a & 0xffff], Y[a >> 16]);
            }
        }
#pragma unroll
        for (int w = 4; w > 0; w >>= 1)
#pragma unroll
            for (int j = 0; j < w; ++j) {
                r[j].x += r[j + w].x;
                r[j].y += r[j + w].y;
            }
#pragma unroll
        for (int w = 16; w > 0; w >>= 1) {
            r[0].x += __shfl_down_sync(0xffffffffu, r[0].x, w);
            r[0].y += __shfl_down_sync(0xffffffffu, r[0].y, w);
        }
        if (lane == 0) *D = r[0];
        return;
    }
    const uint32_t xy = t.xy + lane_strides(lane, op.xy);
    float2 v;
    if (op.kind == SEGOP_COPY) {
        v = X[xy & 0xffff];
    } else {
        const uint32_t klane = lane_strides(lane, op.k);  // the offsets of k = lane (of k's five low bits)
        v = make_float2(0.f, 0.f);
        if (kb == 0) mac<1>(v, X, Y, xy, klane, 0);
        else if (kb == 1) mac<2>(v, X, Y, xy, klane, 0);
        else if (kb == 2) mac<4>(v, X, Y, xy, klane, 0);
        else if (kb <= 5) {
            for (int k = 0; k < 1 << kb; k += 8) mac<8>(v, X, Y, xy, klane, k);
        } else {
            for (int k0 = 0; k0 < 1 << kb; k0 += 64) {  // partial sums of 64 k
                float2 acc = make_float2(0.f, 0.f);
#pragma unroll
                for (int h = 0; h < 64; h += 32) {
                    const uint32_t base = xy + strides((uint32_t)(k0 + h) >> 5, op.k + 5);
                    for (int k = 0; k < 32; k += 8) mac<8>(acc, X, Y, base, klane, k);
                }
                v.x += acc.x;
                v.y += acc.y;
            }
        }
    }
    if (lane < t.n) {
        const uint4 p = *(const uint4*)op.d;  // eight 16-bit offsets
        const uint32_t d = ((lane & 1) ? p.x & 0xffff : 0u) + ((lane & 2) ? p.x >> 16 : 0u) +
                           ((lane & 4) ? p.y & 0xffff : 0u) + ((lane & 8) ? p.y >> 16 : 0u) +
                           ((lane & 16) ? p.z & 0xffff : 0u);
        D[d] = v;
    }
}

__global__ void __launch_bounds__(512) k_seg(const __grid_constant__ SegCtx c) {
    extern __shared__ int4 seg_smem[];
    const uint8_t* src = c.prog + (c.prog_off ? c.prog_off[blockIdx.y] : 0);
    const int bytes = ((const SegHdr*)src)->bytes;
    uint8_t* prog = (uint8_t*)seg_smem;
    float2* arena = (float2*)(prog + c.prog_bytes);
    for (int i = threadIdx.x; i < bytes / 16; i += blockDim.x) ((int4*)prog)[i] = ((const int4*)src)[i];
    __syncthreads();
    const SegHdr& h = *(const SegHdr*)prog;
    auto pad16 = [](size_t b) { return (b + 15) & ~(size_t)15; };
    const SegIn* ins = (const SegIn*)(prog + pad16(sizeof(SegHdr)));
    const SegOp* ops = (const SegOp*)((const uint8_t*)ins + pad16(h.n_in * sizeof(SegIn)));
    const SegTask* tasks = (const SegTask*)((const uint8_t*)ops + pad16(h.n_ops * sizeof(SegOp)));
    const int32_t* bound = (const int32_t*)((const uint8_t*)tasks + pad16(h.n_tasks * sizeof(SegTask)));
    const int warp = threadIdx.x >> 5, warps = blockDim.x >> 5;
    load_inputs(ins, h.n_tiny, h.n_in, c, blockIdx.x, true, arena);
    for (int64_t item = blockIdx.x; item < c.n_items; item += gridDim.x) {
        load_inputs(ins, h.n_tiny, h.n_in, c, item, false, arena);
        float2* result = c.region[h.out_space] + h.out_off * c.cap[h.out_space] + item * h.out_entries;
        __syncthreads();
        for (int s = 0; s < h.n_stages; ++s) {
            for (int t = bound[s] + warp; t < bound[s + 1]; t += warps) run_task(ops[tasks[t].op], tasks[t], arena, result);
            __syncthreads();
        }
    }
}

}  // namespace

cudaError_t launch_seg(const SegCtx& c, int n_progs, int threads, cudaStream_t st) {
    if (c.n_items <= 0 || n_progs <= 0) return cudaSuccess;
    if (c.n_items > kMaxBatchItems) return cudaErrorInvalidValue;
    const int smem = c.prog_bytes + c.arena * (int)sizeof(float2);
    if (smem > kSegMaxSmem) return cudaErrorInvalidValue;
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    static uint64_t done[4] = {0, 0, 0, 0};  // shared-memory opt-in, once per device
    static std::mutex mu;
    int sms = 152;
    {
        std::lock_guard<std::mutex> lk(mu);
        if (dev < 256 && !((done[dev >> 6] >> (dev & 63)) & 1)) {
            e = cudaFuncSetAttribute(k_seg, cudaFuncAttributeMaxDynamicSharedMemorySize, kSegMaxSmem);
            if (e != cudaSuccess) return e;
            done[dev >> 6] |= 1ull << (dev & 63);
        }
    }
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms <= 0) sms = 152;
    // as many CTAs as the SMs hold at once; a CTA keeps its program over the items it walks
    int per_sm = (220 * 1024) / (smem + 1024);
    if (per_sm > 2048 / threads) per_sm = 2048 / threads;
    if (per_sm < 1) per_sm = 1;
    const int64_t fill = (int64_t)sms * per_sm;
    const dim3 grid((unsigned)(c.n_items < fill ? c.n_items : fill), (unsigned)n_progs);
    k_seg<<<grid, threads, smem, st>>>(c);
    return cudaGetLastError();
}

}  // namespace qx
