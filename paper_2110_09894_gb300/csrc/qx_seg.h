// Segments: connected groups of small steps of one dependence level that one launch runs with every
// intermediate in shared memory (k_seg, qx_seg.cu).  Built by the plan compiler (qx_host.cpp).
#pragma once

#include "qx_internal.h"

namespace qx {

constexpr int kSegMaxBits = 12;   // entries of one tensor of a segment: at most 2^12
constexpr int kSegFix = kMaxFix;

// An operand that comes from outside the segment: copied into the arena (compact, leg 0 most
// significant) before the steps run.  once = 1: the same for every item, copied once per CTA.
struct SegIn {
    int64_t off;       // entries from the start of its space (a region's offset is per item: times the capacity)
    int32_t space;     // SEG_LEAF, or the level of its storage region (SEG_INV, SEG_SLICE, SEG_PAIR)
    int32_t rank;
    int32_t arena;     // its entries in the arena
    int32_t once;
    int32_t n_fix;
    int32_t natural;   // entry e sits at off + e
    int32_t fix_src[kSegFix];
    int32_t fix_stride[kSegFix];
    int8_t pos[kSegMaxBits];  // address position of entry bit b (0 = least significant)
    int32_t pad;
};
enum { SEG_INV = 0, SEG_SLICE = 1, SEG_PAIR = 2, SEG_LEAF = 3 };

// One step: out[d(o)] = sum_k X[x(o) + xk(k)] Y[y(o) + yk(k)] over the natural output index o (columns
// low, then rows).  Offsets add up over the set bits; an offset pair holds X's entry offset in its low
// 16 bits and Y's in its high ones.  A task covers 32 outputs, so the step keeps the pairs (xy) and
// result offsets (d) of the five low output bits only.
struct alignas(16) SegOp {
    int32_t kind;          // SEGOP_MAC, SEGOP_COPY (Y unused) or SEGOP_DOT (256 strided partials, then a tree)
    int32_t kb;            // contracted bits
    int32_t x, y;          // arena entries
    int32_t dst;           // arena entry; < 0: the segment's result, written to its storage
    int32_t pad[3];
    uint32_t xy[8];        // output bits 0 .. 4
    uint32_t k[kSegMaxBits];
    uint16_t d[8];         // output bits 0 .. 4
};
enum { SEGOP_MAC = 0, SEGOP_COPY = 1, SEGOP_DOT = 2 };

// Work of one warp: n <= 32 outputs of a step (a dot product: one), from output o0 on, whose offset
// pair and result offset are xy and d.  Tasks of one stage touch no common result; a block barrier
// separates the stages.
struct alignas(16) SegTask {
    int32_t op, n;
    uint32_t xy, d;
};

// One segment's program: the header, then n_in SegIn, n_ops SegOp, n_tasks SegTask and
// n_stages + 1 int32 task bounds, each array 16-byte aligned.
struct SegHdr {
    int32_t n_in, n_ops, n_tasks, n_stages;
    int32_t n_tiny;        // leading operands of at most 16 entries
    int32_t pad0;
    int32_t bytes;         // of the whole program, a multiple of 16
    int32_t arena;         // entries
    int32_t out_space;     // region of the result
    int32_t out_entries;
    int64_t out_off;
};

struct SegCtx {
    const uint8_t* prog;       // device: programs, program c at prog_off[c] (n_progs > 1) or prog
    const int32_t* prog_off;   // device
    const float2* leaves;
    float2* region[3];         // invariant, per-slice and per-pair region
    int64_t cap[3];            // items the regions have room for (1 for the invariant one)
    int64_t n_items;           // items of this launch
    int32_t per_pair;          // items are (slice, bitstring) pairs: a per-slice operand is item / n_b
    int32_t prog_bytes, arena; // shared memory: the largest program, the largest arena
    ItemCtx ic;
};
cudaError_t launch_seg(const SegCtx& c, int n_progs, int threads, cudaStream_t st);
constexpr int kSegMaxSmem = 200 * 1024;

}  // namespace qx
