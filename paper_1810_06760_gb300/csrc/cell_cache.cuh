// Model sampling through a per-thread copy of the current grid cell (FP32 path).
//
// The trilinear interpolation of the 10 fields reads 8 nodes of 48 bytes.  Beams of a warp sit in different cells,
// so read straight from global memory those 24 16-byte loads touch up to 32 lines each and the L1 data pipe bounds
// the RK4 kernel (409 wavefronts per warp and right-hand side, the pipe 80% busy).  A beam stays in a cell for
// several right-hand sides (dt c is a fraction of a cell, and two of the four RK4 stages share the position to
// O(dt^2)), so every thread keeps its cell's four rows of two nodes in a column of shared memory and refills
// it by cp.async only when the cell changes.  The position of the next right-hand side is known early in the
// current one, so the copies are in flight while it is finished.
//
// Columns are 25 float4 apart, so that a quarter warp's 16-byte reads of one chunk fall into distinct banks.
// A warp filling its lanes' cells together (24 lanes a cell, whole lines at a time) took fewer wavefronts but
// ten instructions per cell: 74.7 against 65.2 ms of propagation on 2.7 M beams x 200 steps.
#pragma once

#include "fga_beam.cuh"

namespace fga {

constexpr int CELL_STRIDE = 25;   // float4 per thread

struct CellCache {
    const float4 *grid;
    const float4 *col;       // this thread's column
    uint32_t cell;           // node index of the lower corner held in the column
    float fr[3];             // fractions of the position last prefetched

    __device__ __forceinline__ void init(const float4 *G, const float4 *smem) {
        grid = G;
        col = smem + (size_t)threadIdx.x * CELL_STRIDE;
        cell = 0xffffffffu;
    }
    // the cell of x and its fractions; starts the copies if the cell changed (after the column has been read)
    __device__ __forceinline__ void prefetch(const ModelDev &M, const float x[3]) {
        int i[3];
#pragma unroll
        for (int d = 0; d < 3; d++) {
            float t = (x[d] - M.fo[d]) * M.finv_h[d];
            const float hi = (float)(M.n[d] - 1);
            t = t < 0.f ? 0.f : (t > hi ? hi : t);
            int id = (int)floorf(t);
            id = id > M.n[d] - 2 ? M.n[d] - 2 : id;
            i[d] = id;
            fr[d] = t - (float)id;
        }
        const uint32_t c = ((uint32_t)i[0] * (uint32_t)M.n[1] + (uint32_t)i[1]) * (uint32_t)M.n[2] + (uint32_t)i[2];
        if (c != cell) {
            const int64_t s1 = 3 * (int64_t)M.n[2], s0 = s1 * M.n[1];
            const float4 *g = grid + 3 * (uint64_t)c;
            const uint32_t sa = (uint32_t)__cvta_generic_to_shared(col);
#pragma unroll
            for (int r = 0; r < 4; r++) {
                const float4 *gr = g + (r >> 1) * s0 + (r & 1) * s1;
#pragma unroll
                for (int k = 0; k < 6; k++)
                    if (k % 3 < 2)
                        asm volatile("cp.async.ca.shared.global [%0], [%1], 16;" ::"r"(sa + (6 * r + k) * 16), "l"(gr + k) : "memory");
                    else
                        asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(sa + (6 * r + k) * 16), "l"(gr + k) : "memory");
            }
        }
        cell = c;
        asm volatile("cp.async.commit_group;" ::: "memory");
    }
    // the 10 fields at the position last prefetched
    __device__ __forceinline__ void sample(float cf[10]) const {
        asm volatile("cp.async.wait_group 0;" ::: "memory");
        const float a1 = fr[0], a0 = 1.0f - a1, b1 = fr[1], b0 = 1.0f - b1, c1 = fr[2], c0 = 1.0f - c1;
        const float ab[4] = {a0 * b0, a0 * b1, a1 * b0, a1 * b1};
        float2 acc[5];
#pragma unroll
        for (int r = 0; r < 4; r++) {
#pragma unroll
            for (int k = 0; k < 2; k++) {
                const float w = ab[r] * (k ? c1 : c0);
                const float2 w2 = make_float2(w, w);
                const float4 *p = col + 6 * r + 3 * k;
                const float4 u0 = p[0], u1 = p[1];
                const float2 u2 = *reinterpret_cast<const float2 *>(p + 2);
                const float2 v[5] = {make_float2(u0.x, u0.y), make_float2(u0.z, u0.w), make_float2(u1.x, u1.y),
                                     make_float2(u1.z, u1.w), u2};
#pragma unroll
                for (int f = 0; f < 5; f++)
                    acc[f] = (r == 0 && k == 0) ? __fmul2_rn(w2, v[f]) : __ffma2_rn(w2, v[f], acc[f]);
            }
        }
#pragma unroll
        for (int f = 0; f < 5; f++) {
            cf[2 * f] = acc[f].x;
            cf[2 * f + 1] = acc[f].y;
        }
    }
};

}  // namespace fga
