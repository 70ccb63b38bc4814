// Uniform hashed cell grid shared by the bond builder and the contact search.
//
// A node at p falls in the integer cell c = floor((p - lo) / cs) (FP64), clamped
// to +-2^20 cells per axis.  Cells hash into a power-of-two bucket table; the nodes are
// counted into the buckets (a counting sort whose order inside a bucket and of the
// buckets is arbitrary) with copies of their cells and FP32 positions, and a query walks
// the 27 cells around a node, keeping only nodes whose own cell is the visited cell.
// The exact distance predicate is applied by the caller, who also orders what it finds,
// so hashing, clamping and the order never change a result.
#pragma once

#include "pd_internal.cuh"

struct GridView {
    double lo[3];
    double inv;                   // 1 / cell size
    uint32_t mask;                // bucket table size - 1
    const uint2 *range;           // bucket -> first entry, one past last
    const uint32_t *node;         // entry -> node index
    const uint64_t *ecell;        // entry -> packed cell coordinates
    const float4 *epf;            // entry -> FP32 position (as pf)
    const uint64_t *cell;         // node -> packed cell coordinates
    const float4 *pf;             // node -> FP32 (p - lo), .w = max |component| (prefilter)
};

// Device buffers of the grid: n entries or nodes each, nbuckets counts and ranges.  The
// two cursors follow the counts, so that one memset clears them all.
struct GridBuf {
    uint32_t nbuckets;
    uint32_t *count;              // nbuckets + 4 words
    uint2 *range;
    uint32_t *key, *rank, *node;
    uint64_t *cell, *ecell;
    float4 *pf, *epf;
    unsigned *bucket_cursor() const { return count + nbuckets; }
    unsigned long long *cand_cursor() const { return (unsigned long long *)(count + nbuckets + 2); }
};

// Conservative FP32 distance test.  pf = fl32(p - lo) carries an error of at
// most 2^-24 |pf|_inf per component; a difference of two such points and its
// squared norm in FP32 stay within r + 1.04e-7 (m_i + m_j) + 1.5e-7 r of the
// exact distance r (m = max |component|).  The bound below is four times that.
__device__ __forceinline__ float pf_slack(float cut, const float4 &a, const float4 &b)
{
    return cut * 1e-6f + 4e-7f * (a.w + b.w);
}
__device__ __forceinline__ float pf_dist2(const float4 &a, const float4 &b)
{
    const float dx = b.x - a.x, dy = b.y - a.y, dz = b.z - a.z;
    return fmaf(dx, dx, fmaf(dy, dy, dz * dz));
}

// (p - lo) / cs rounds to within 2^-31 of a cell over the clamped range, far below the
// 1e-7 by which every cell is wider than its search distance
__device__ __forceinline__ int grid_coord(double p, double lo, double inv)
{
    return min(max(__double2int_rd(__dmul_rn(__dsub_rn(p, lo), inv)), -1048576), 1048575);
}

__device__ __forceinline__ uint64_t grid_pack(int cx, int cy, int cz)
{
    return ((uint64_t)((uint32_t)(cx + 1048576) & 0x1fffffu) << 42) |
           ((uint64_t)((uint32_t)(cy + 1048576) & 0x1fffffu) << 21) |
           (uint64_t)((uint32_t)(cz + 1048576) & 0x1fffffu);
}

__device__ __forceinline__ uint32_t grid_hash(int cx, int cy, int cz, uint32_t mask)
{
    return (((uint32_t)cx * 73856093u) ^ ((uint32_t)cy * 19349663u) ^ ((uint32_t)cz * 83492791u)) & mask;
}

// Buckets the nodes at x4 + u: u as FP64 (u4), as double-float pairs (hi, lo, element
// stride `stride`), or none.  Clears both cursors.
void grid_build(GridView &g, const GridBuf &w, const dbl4 *x4, const dbl4 *u4, const float4 *hi, const float4 *lo,
                int stride, int64_t n, double cs, cudaStream_t st);
