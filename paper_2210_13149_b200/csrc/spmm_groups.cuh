// What the aggregations share that take a matrix in groups of stored entries (spmm_bits.cu, spmm_bytes.cu): how the entries are
// split, the range of their weights in fixed point, operands in shared memory; and the stream of groups of a warp.
#pragma once
#include <stdint.h>

#include <cuda_runtime.h>

namespace bigcn {
namespace groups {

constexpr int kGroup = 128;                         // stored entries of a group
constexpr int kRowCost = 4;                         // what a row counts beside its entries where work is split
enum Flags : int { kPair = 1, kDirect = 2, kFirst = 4, kLast = 8, kStarts = 16, kWhole = 32 };

// How the stored entries of a graph are split, made by launch_spmm_bits_plan().
struct GraphPlan {
    int chunk_log2;                                 // entries + kRowCost per row and unit of work
    int chunks;                                     // units
    const int4* groups;                             // of all units: first entry, first row, entries | those of the first row << 8 | Flags << 16
    const int2* units;                              // per unit: its first group, how many
};

// Biased exponents of a largest weight (or sum of weights) that have a fixed point here.
constexpr uint32_t kExpLow = 40, kExpHigh = 230;
constexpr uint32_t kFlip = 0x80808080u;             // (v + kFlip) ^ kFlip: the balanced digits of v, one per byte

// Two 16 x 16 byte matrices, transposed: lane 4 g + t gets byte g (r[0]) and byte g + 8 (r[1]) of rows 4 t .. 4 t + 3 of the
// first, r[2] and r[3] of the second; lane l gives the address of row l of the 32.
__device__ __forceinline__ void ldmatrix_bytes(uint32_t saddr, uint32_t (&r)[4])
{
    asm volatile("ldmatrix.sync.aligned.m16n16.x2.trans.shared.b8 {%0,%1,%2,%3}, [%4];\n"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(saddr) : "memory");
}

// The same value in every lane, known as such to the compiler: it decides branches on it for the warp.
__device__ __forceinline__ int uniform(int v) { return __shfl_sync(0xffffffffu, v, 0); }

// The groups of a warp's units of work, one after the other, with the column indices and values of their entries; a group is
// asked for one ahead.  (agg_bits_kernel, at its limit of registers, has a walk of its own: a unit there is one slice of columns of a
// unit here, and it holds the column indices and values of one group, this struct those of a second beside the caller's.)
struct Stream {
    int unit, step;                                 // the unit after the one at hand; warps of the grid
    int where;                                      // the unit at hand
    int left = 0;                                   // its groups from the one asked for on
    const int4* at;                                 // the group after the one asked for
    int4 asked;
    int first, row, meta, place;                    // the group at hand: its entry in GraphPlan::groups, `where`
    int col[4];                                     // entry 32 i + lane
    float val[4];
    __device__ __forceinline__ Stream(int unit_, int step_) : unit(unit_), step(step_) {}
    __device__ __forceinline__ bool next(const GraphPlan& pl)
    {
        while (left == 0) {
            if (unit >= pl.chunks) return false;
            where = unit;
            const int2 u = __ldg(pl.units + where);
            at = pl.groups + uniform(u.x);
            left = uniform(u.y);
            if (left > 0) asked = __ldg(at++);
            unit += step;
        }
        first = uniform(asked.x);
        row = uniform(asked.y);
        meta = uniform(asked.z);
        place = where;
        if (--left > 0) asked = __ldg(at++);
        return true;
    }
    __device__ __forceinline__ void load(const int32_t* colidx, const float* value, int lane)
    {
        const int cnt = meta & 255;
        // (lanes past the group's end take its last entry with weight 0: a column of their own choice, node 0 say, would send
        // every warp of the GPU to one sector of the L2)
        const int32_t* pc = colidx + first;
        const float* pv = value + first + lane;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            col[i] = 0;
            val[i] = 0.f;
            if (32 * i < cnt) col[i] = __ldg(pc + min(32 * i + lane, cnt - 1));
            if (32 * i + lane < cnt) val[i] = __ldg(pv + 32 * i);
        }
    }
};

}  // namespace groups

groups::GraphPlan spmm_bits_plan_at(int64_t n, int64_t nnz, const void* plan);

}  // namespace bigcn
