// A6 on single-plane lattices (receiver arrays: n0 x n1 points at one x3), FP32 path, on the
// tensor cores with warp-specialised producers.
//
// On a tile of T0 x T1 points of the plane, with E_d the per-axis Gaussian factors of Eq. FGA,
//
//   U[(j,c)][i] = sum_b  W_bc E1_b(x_j) E0_b(x_i),      W_bc = A_bc E2_b(x_2)
//
// is a complex matrix product over the beams b (the contraction index).  One operand B' = [Re E0; Im E0] serves
// both halves of the complex product: A_re B'^T and A_im B'^T (A = W E1) go to two halves of the accumulator, and
// Re U = A_re Re E0 - A_im Im E0, Im U = A_re Im E0 + A_im Re E0 are formed by the reduction over the items.  Both
// operands are FP16 hi/lo splits of the FP32 values (hi*hi + hi*lo + lo*hi, FP32 accumulation): one tcgen05.mma of
// M = 128 ([B'_hi; B'_lo], 64 rows each) x N = 256 (A_re hi, A_re lo, A_im hi, A_im lo, 64 rows each) x K = 16
// beams forms every product (and an unused lo*lo quarter).
//
// One launch takes all samples of a window (work = sample x item), one persistent CTA per SM: three groups of four
// producer warps, 4 epilogue warps and one MMA warp.
//  - Each producer group owns one shared-memory stage of 64 beams.  It filters its share of an item's candidate
//    records (the beams within the window radius of the tile's box; chunks of 128, the next one in flight) into a
//    queue and turns every 64 kept beams into one operand block, 16 beams a warp: lane (h, p) takes beams 2p and
//    2p+1 of the 16 and the quarter h of the points of each axis, forms W, E1 and E0 by recurrence along its
//    quarters, in packed FP32x2 registers (beam 2p, beam 2p+1), waits for the stage and writes pairs of FP16
//    values straight into the K-major operands.  The rows of the quarters are interleaved (row 4 n + h holds
//    point n of quarter h), so that the four quarters' stores of an instruction fill 128 contiguous bytes of the
//    32-byte-swizzled layout: no bank conflicts and no padding (core matrices padded to 144 bytes against the
//    conflicts made the tensor cores read two lines for one).
//  - Per stage a "full" mbarrier (producers -> MMA) and an "empty" one (tcgen05.commit -> producers).  With one
//    stage per group every parity wait is exactly one phase behind the barrier.
//  - The MMA warp's elected thread takes the groups' blocks in a fixed cyclic order (so the accumulation order, and
//    the result, do not depend on timing), four MMAs and one commit each.  Its serial chain per block (wait,
//    header, commit: 400 cycles besides the MMAs) set the pace when every 16 or 32 beams were a block.
//  - A group's last block of an item is marked; when every group has sent it, the accumulator (one of two, 256
//    columns each) is handed to the epilogue warps, which copy it to the item's partial sums while the next item
//    accumulates in the other one.
// What bounds it: the producers' issue slots (860 warp instructions per 16 beams and 378 cycles of an SM; on 0.44 M beams
// and one window of samples of 16 x 16 receivers 58% of the slots, tensor pipe 30%, shared memory 39%).  Sums of a solve, against one launch per sample with
// seven single-warp producers and padded operands: 200 samples of 2.7 M beams on 16 x 16 receivers 48.7 -> 26.9 ms
// (0.44 M beams: 13.4 -> 5.7 ms), 250 samples of 8.4 M beams on 20 x 20 receivers 192 -> 118 ms; the reductions
// 4.9 -> 1.0, 3.3 -> 0.5 and 7.1 -> 3.2 ms.
// Every wait is bounded: a wait that runs out sets the call's error word, which ends the other waits of the launch;
// the producers then run through their barrier schedule without waiting or writing, the other roles leave their
// loops, the MMA thread waits (bounded) for its outstanding MMAs, and the tensor memory is freed.
#include <algorithm>
#include <cmath>

#include "fga_beam.cuh"
#include "gather.cuh"
#include "tcgen05.cuh"

namespace fga {

// in-window pairs counted by the counting instantiation (profiling)
static __device__ unsigned long long g_plane_pairs;

int64_t read_plane_pair_counter(bool reset) {
    unsigned long long v = 0;
    if (cudaMemcpyFromSymbol(&v, g_plane_pairs, sizeof v) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    if (reset) {
        const unsigned long long z = 0;
        cudaMemcpyToSymbol(g_plane_pairs, &z, sizeof z);
    }
    return (int64_t)v;
}

namespace {

constexpr int PL_GROUPS = 3;                   // producer groups, one shared-memory stage each
constexpr int PL_GW = 4;                       // warps of a group
constexpr int PL_PROD = PL_GROUPS * PL_GW;     // producer warps
constexpr int PL_EPI = 4;                      // epilogue warps, one per quadrant of the TMEM lanes
constexpr int PL_WARPS = PL_PROD + PL_EPI + 1; // + the MMA warp
constexpr int PL_THREADS = PL_WARPS * 32;
constexpr int PL_KB = 16;                      // beams per MMA
constexpr int PL_BLOCK = PL_GW * PL_KB;        // beams per block
constexpr int PL_ROW = 2 * PL_KB;              // bytes of an operand row
constexpr int PL_COPY = 64 * PL_ROW;           // one operand copy: 64 rows
constexpr int PL_OPS = 6 * PL_COPY;            // A_re hi, A_re lo, A_im hi, A_im lo, B' hi, B' lo of 16 beams
constexpr int PL_STAGE = PL_GW * PL_OPS;
constexpr int PL_QUEUE = 256;                  // kept records queued per group (63 + 128 used)
constexpr int PL_LAST = 1 << 16;               // header flag: the group's last block of the item
constexpr int PL_T0_MAX = 24, PL_T1_MAX = 20;  // 6 points and 5 rows (15 operand rows) per quarter
constexpr int PL_SMEM = PL_GROUPS * (PL_STAGE + PL_QUEUE * 48) + 512 + 1024;   // 1 KB to align the stages
constexpr uint32_t PL_ACC = 256;               // accumulator columns (two accumulators)


struct PlaneArgs {
    const float *rec;        // records [sample][n_rec][12]: Q, P, weighted polarised amplitude (3 complex)
    int64_t rec_stride;      // floats between samples
    const int4 *items;       // (tile, first record, end record, 0)
    int nitems, nwork;       // work = sample * nitems + item (items of the launch's tiles)
    int n0, n1;              // lattice extents (n2 = 1)
    int T0, T1, nt1;         // tile shape and tiles along axis 1
    float x0, h0, x1, h1, x2;  // uniform axes 0 and 1, the plane's x3
    float k, rw2;
    const float *amax;       // per sample: bound of |A| over the records
    float *partial;          // [work][re, im of A][12 ceil(T1/4) columns][128 lanes]
    int *err;
};

// FP16 hi/lo split of a packed pair, as two f16x2 words, the residual by one packed subtraction
__device__ __forceinline__ void split2p(float2 v, uint32_t &hi, uint32_t &lo) {
    const __half2 hh = __float22half2_rn(v);
    const float2 hf = __half22float2(hh);
    const __half2 ll = __float22half2_rn(__fadd2_rn(v, make_float2(-hf.x, -hf.y)));
    hi = *reinterpret_cast<const uint32_t *>(&hh);
    lo = *reinterpret_cast<const uint32_t *>(&ll);
}

__device__ __forceinline__ void sts32(unsigned char *base, uint32_t off, uint32_t v) {
    *reinterpret_cast<uint32_t *>(base + off) = v;
}

// bounded wait (2^22 polls; the stages turn over in microseconds, an item in less than a second), which also
// gives up once any CTA of the launch has reported a timeout in the call's error word
__device__ __forceinline__ bool bar_wait(uint32_t bar, uint32_t parity, const int *gerr) {
    for (int it = 0; it < (1 << 22); it++) {
        uint32_t ready;
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}"
            : "=r"(ready)
            : "r"(bar), "r"(parity)
            : "memory");
        if (ready) return true;
        if ((it & 1023) == 1023 && *reinterpret_cast<const volatile int *>(gerr) != 0) return false;
    }
    return false;
}

__device__ __forceinline__ void bar_arrive(uint32_t bar) {
    asm volatile("mbarrier.arrive.release.cta.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}

// first wait of a launch that gave up: the error word plus where (1 producer stage wait, 3 MMA wait for a
// block, 4 MMA wait for a free accumulator, 5 epilogue wait), the block, its stage and parity, the blocks
// claimed and the CTA (words 2..7 of the call's status words)
__device__ __forceinline__ void report_timeout(int *err, int site, int n, int s, int parity, int claimed, int consumed) {
    atomicExch(err, 1);
    if (atomicCAS(err + 2, 0, site) == 0) {
        err[3] = n;
        err[4] = s;
        err[5] = parity;
        err[6] = claimed;
        err[7] = blockIdx.x;
        err[8] = consumed;
    }
}

// power-of-two scale of the amplitude operand for a bound of the amplitudes: |A| * scale <= 2^14
__device__ __forceinline__ float plane_scale(float bound) {
    float sa = 1.0f;
    if (bound > 0.0f && isfinite(bound)) {
        int e;
        frexpf(bound, &e);
        sa = ldexpf(1.0f, 14 - e);
    }
    return sa;
}
constexpr float PL_SB = 16384.0f;   // scale of the E0 operand

// a complex value of each of the lane's two beams: real parts and imaginary parts as packed pairs
struct Pair {
    float2 r, i;
    __device__ __forceinline__ Pair mul(const Pair &o) const {
        return {__ffma2_rn(make_float2(-i.x, -i.y), o.i, __fmul2_rn(r, o.r)), __ffma2_rn(i, o.r, __fmul2_rn(r, o.i))};
    }
    __device__ __forceinline__ void scale(float2 g) {
        r = __fmul2_rn(r, g);
        i = __fmul2_rn(i, g);
    }
};

// JT, IT: rows j and points i per quarter as compile-time constants (the loops unroll, operand offsets become
// immediates); 0 = taken from the launch
template <bool COUNT, int JT, int IT>
__global__ void __launch_bounds__(PL_THREADS, 1) plane_tc_kernel(PlaneArgs P) {
    extern __shared__ unsigned char smem_raw[];
    unsigned char *smem = smem_raw + ((1024 - (tc::smem_u32(smem_raw) & 1023)) & 1023);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    float4 *queues = reinterpret_cast<float4 *>(smem + PL_GROUPS * PL_STAGE);   // [PL_GROUPS][PL_QUEUE][3]
    unsigned char *tail = smem + PL_GROUPS * (PL_STAGE + PL_QUEUE * 48);
    int4 *counts = reinterpret_cast<int4 *>(tail);          // [PL_GROUPS][2]: kept records of a chunk per warp
    uint64_t *full = reinterpret_cast<uint64_t *>(counts + 2 * PL_GROUPS);
    uint64_t *empty = full + PL_GROUPS;
    uint64_t *accfull = empty + PL_GROUPS;  // [2] an accumulator is complete (commit + the MMA thread)
    uint64_t *accfree = accfull + 2;        // [2] its epilogue is done (four warps)
    uint64_t *done = accfree + 2;
    int *hdr = reinterpret_cast<int *>(done + 1);          // per stage: beams in the block, with PL_LAST
    int *have = hdr + PL_GROUPS;                           // [2] the accumulator received an MMA
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(have + 2);

    if (warp == PL_WARPS - 1) tc::alloc(tc::smem_u32(tmem_slot), 2 * PL_ACC);
    if (tid == 0) {
        for (int s = 0; s < PL_GROUPS; s++) {
            tc::mbar_init_n(tc::smem_u32(full + s), PL_GW);
            tc::mbar_init(tc::smem_u32(empty + s));
        }
        for (int a = 0; a < 2; a++) {
            tc::mbar_init_n(tc::smem_u32(accfull + a), 2);
            tc::mbar_init_n(tc::smem_u32(accfree + a), PL_EPI);
        }
        tc::mbar_init(tc::smem_u32(done));
    }
    tc::fence_before();
    __syncthreads();
    tc::fence_after();
    const uint32_t tmem = *tmem_slot;

    const int J = JT ? JT : (P.T1 + 3) >> 2;         // rows j per quarter
    const int I = IT ? IT : (P.T0 + 3) >> 2;         // points i per quarter
    const int MI = (4 * I + 7) / 8 * 8;              // first Im row of B'
    const int ncol = 12 * J;                         // operand rows of A in use

    if (warp < PL_PROD) {
        // ------------------------------------------------ producers ------------------------------------
        const int g = warp / PL_GW, wg = warp % PL_GW;
        float4 *q = queues + g * PL_QUEUE * 3;
        const int h = lane >> 3, p = lane & 7;
        unsigned char *st = smem + g * PL_STAGE + wg * PL_OPS;
        // row 4 n + h, beams 2p, 2p+1: 128 n + 32 h + the 16-byte half (exchanged for odd n) + 4 (p & 3)
        const uint32_t off_even = (uint32_t)(h * 32 + ((p >> 2) << 4) + (p & 3) * 4), off_odd = off_even ^ 16u;
        const float hk = -0.5f * P.k;
        const float g1 = __expf(-P.k * P.h1 * P.h1), g0 = __expf(-P.k * P.h0 * P.h0);
        const float2 G1 = make_float2(g1, g1), G0 = make_float2(g0, g0);
        unsigned long long pairs = 0;
        int uses = 0;   // blocks of the stage so far
        bool ok = true;
        // wait until the MMAs of this stage's previous block are done (exactly one phase back)
        auto acquire = [&]() {
            if (uses > 0 && ok) {
                bool wt = true;
                if (lane == 0) {
                    wt = bar_wait(tc::smem_u32(empty + g), (uint32_t)((uses - 1) & 1), P.err);
                    if (!wt) report_timeout(P.err, 1, uses, g, (uses - 1) & 1, uses, 0);
                }
                ok = __shfl_sync(0xffffffffu, wt ? 1 : 0, 0) != 0;
            }
        };
        auto release = [&](int value) {
            __syncwarp();
            if (lane == 0) {
                if (wg == 0) hdr[g] = value;
                bar_arrive(tc::smem_u32(full + g));
            }
            uses++;
        };
        auto group_sync = [&]() { asm volatile("bar.sync %0, %1;" ::"r"(1 + g), "n"(PL_GW * 32) : "memory"); };
        int par = 0;    // half of the group's counters for the next chunk
        for (int work = blockIdx.x; work < P.nwork; work += gridDim.x) {
            const int item = work % P.nitems, samp = work / P.nitems;
            const int4 it = P.items[item];
            const int t = it.x, tt0 = t / P.nt1, tt1 = t % P.nt1;
            const int i0 = tt0 * P.T0, j0 = tt1 * P.T1;
            const int e0 = min(P.T0, P.n0 - i0), e1 = min(P.T1, P.n1 - j0);
            const float *rec = P.rec + samp * P.rec_stride;
            const float sa = plane_scale(P.amax[samp]);
            // the tile's box (window test of the candidates)
            const float blo0 = P.x0 + P.h0 * i0, bhi0 = P.x0 + P.h0 * (i0 + e0 - 1);
            const float blo1 = P.x1 + P.h1 * j0, bhi1 = P.x1 + P.h1 * (j0 + e1 - 1);
            const float xq0 = P.x0 + P.h0 * (float)(i0 + h * I), xq1 = P.x1 + P.h1 * (float)(j0 + h * J);
            int qh = 0, qt = 0;
            auto produce = [&](int nblock, int flag) {
                const int nvalid = min(PL_KB, nblock - PL_KB * wg);   // this warp's beams of the block
                if (nvalid <= 0) {
                    acquire();
                    release(nblock | flag);
                    return;
                }
                // factors of the lane's two beams, in registers, before the stage is needed
                Pair W[3], F1, R1, F0, R0;
#pragma unroll
                for (int u = 0; u < 2; u++) {
                    const int slot = 2 * p + u;
                    float r[REC];
                    if (slot < nvalid) {
                        const float4 *src = q + ((qh + PL_KB * wg + slot) & (PL_QUEUE - 1)) * 3;
                        const float4 a = src[0], b = src[1], c = src[2];
                        r[0] = a.x; r[1] = a.y; r[2] = a.z; r[3] = a.w;
                        r[4] = b.x; r[5] = b.y; r[6] = b.z; r[7] = b.w;
                        r[8] = c.x; r[9] = c.y; r[10] = c.z; r[11] = c.w;
                    } else {   // padding: a beam of zero amplitude in the tile (finite factors)
#pragma unroll
                        for (int f = 3; f < REC; f++) r[f] = 0.f;
                        r[0] = blo0;
                        r[1] = blo1;
                        r[2] = P.x2;
                    }
                    auto put = [&](Pair &v, float re, float im) {
                        if (u == 0) {
                            v.r.x = re;
                            v.i.x = im;
                        } else {
                            v.r.y = re;
                            v.i.y = im;
                        }
                    };
                    // W_c = A_c E2 (scaled for the A operand); zero for padding beams
                    float er, ei;
                    const float dz = P.x2 - r[2];
                    gauss_phase_exp<float>(P.k * r[5] * dz, hk * dz * dz, &er, &ei);
                    const float scl = slot < nvalid ? sa : 0.f;
#pragma unroll
                    for (int c = 0; c < 3; c++)
                        put(W[c], scl * (r[6 + 2 * c] * er - r[7 + 2 * c] * ei),
                            scl * (r[6 + 2 * c] * ei + r[7 + 2 * c] * er));
                    // E1, E0 at the first point of the lane's quarters, and their ratios for one step
                    const float d1 = xq1 - r[1], d0 = xq0 - r[0];
                    gauss_phase_exp<float>(P.k * r[4] * d1, hk * d1 * d1, &er, &ei);
                    put(F1, er, ei);
                    gauss_phase_exp<float>(P.k * r[3] * d0, hk * d0 * d0, &er, &ei);
                    const float sb = slot < nvalid ? PL_SB : 0.f;
                    put(F0, sb * er, sb * ei);
                    if (J > 1) {
                        gauss_phase_exp<float>(P.k * r[4] * P.h1, -P.k * P.h1 * (d1 + 0.5f * P.h1), &er, &ei);
                        put(R1, er, ei);
                    }
                    if (I > 1) {
                        gauss_phase_exp<float>(P.k * r[3] * P.h0, -P.k * P.h0 * (d0 + 0.5f * P.h0), &er, &ei);
                        put(R0, er, ei);
                    }
                    if (COUNT && slot < nvalid) {
                        // pairs of this beam inside the window, rows of this quarter
                        const float dz2 = dz * dz;
                        for (int jj = h * J; jj < min(e1, (h + 1) * J); jj++) {
                            const float dy = P.x1 + P.h1 * (float)(j0 + jj) - r[1];
                            const float s2 = P.rw2 - dz2 - dy * dy;
                            if (s2 < 0.f) continue;
                            const float sq = sqrtf(s2);
                            if (P.h0 > 0.f) {
                                const int lo = max(0, (int)ceilf((r[0] - sq - blo0) / P.h0));
                                const int hi = min(e0 - 1, (int)floorf((r[0] + sq - blo0) / P.h0));
                                if (hi >= lo) pairs += (unsigned long long)(hi - lo + 1);
                            } else if (fabsf(r[0] - blo0) <= sq) {
                                pairs += 1ull;
                            }
                        }
                    }
                }
                acquire();
                if (ok) {
                    unsigned char *B = st + 4 * PL_COPY;
#pragma unroll
                    for (int t1 = 0; t1 < (JT ? JT : J); t1++) {
#pragma unroll
                        for (int c = 0; c < 3; c++) {
                            const int n = 3 * t1 + c;
                            const Pair v = W[c].mul(F1);
                            uint32_t rh, rl, ih, il;
                            split2p(v.r, rh, rl);
                            split2p(v.i, ih, il);
                            const uint32_t o = (uint32_t)(n * 128) + ((n & 1) ? off_odd : off_even);
                            sts32(st, o, rh);
                            sts32(st + PL_COPY, o, rl);
                            sts32(st + 2 * PL_COPY, o, ih);
                            sts32(st + 3 * PL_COPY, o, il);
                        }
                        if (t1 + 1 < (JT ? JT : J)) {
                            F1 = F1.mul(R1);
                            R1.scale(G1);
                        }
                    }
#pragma unroll
                    for (int n = 0; n < (IT ? IT : I); n++) {
                        uint32_t rh, rl, ih, il;
                        split2p(F0.r, rh, rl);
                        split2p(F0.i, ih, il);
                        const uint32_t o = (uint32_t)(n * 128) + ((n & 1) ? off_odd : off_even);
                        const uint32_t oi = o + (uint32_t)(MI * PL_ROW);
                        sts32(B, o, rh);
                        sts32(B + PL_COPY, o, rl);
                        sts32(B, oi, ih);
                        sts32(B + PL_COPY, oi, il);
                        if (n + 1 < (IT ? IT : I)) {
                            F0 = F0.mul(R0);
                            R0.scale(G0);
                        }
                    }
                    // make the stores visible to the tensor cores, then hand the stage over
                    tc::fence_async_smem();
                }
                release(nblock | flag);
            };
            // candidates of this group: chunks of 128 records dealt round robin over the groups; the next chunk's
            // records are loaded (coalesced, one record per lane) while this one is filtered and its kept records
            // are queued in shared memory and turned into blocks
            const int64_t stride = 32 * PL_PROD;
            const int64_t mine = 32 * wg + lane;
            int64_t c0 = (int64_t)it.y + 128 * g;
            float4 na = make_float4(0.f, 0.f, 0.f, 0.f), nb = na, nc = na;
            if (c0 + mine < it.z) {
                const float4 *src = reinterpret_cast<const float4 *>(rec + (c0 + mine) * REC);
                na = src[0];
                nb = src[1];
                nc = src[2];
            }
            for (; c0 < it.z; c0 += stride) {
                const float4 ra = na, rb = nb, rc = nc;
                const int64_t c = c0 + mine, cn = c + stride;
                if (cn < it.z) {
                    const float4 *src = reinterpret_cast<const float4 *>(rec + cn * REC);
                    na = src[0];
                    nb = src[1];
                    nc = src[2];
                }
                bool kp = false;
                if (c < it.z) {
                    const float g0d = fmaxf(fmaxf(blo0 - ra.x, ra.x - bhi0), 0.f);
                    const float g1d = fmaxf(fmaxf(blo1 - ra.y, ra.y - bhi1), 0.f);
                    const float g2d = P.x2 - ra.z;
                    kp = g0d * g0d + g1d * g1d + g2d * g2d <= P.rw2;
                }
                const unsigned bl = __ballot_sync(0xffffffffu, kp);
                int4 *cnt = counts + 2 * g + par;
                par ^= 1;
                if (lane == 0) reinterpret_cast<int *>(cnt)[wg] = __popc(bl);
                group_sync();   // the counts; and every warp is done with the blocks before (their queue slots)
                const int4 n4 = *cnt;
                const int before = (wg > 0 ? n4.x : 0) + (wg > 1 ? n4.y : 0) + (wg > 2 ? n4.z : 0);
                if (kp) {
                    float4 *dst = q + ((qt + before + __popc(bl & ((1u << lane) - 1u))) & (PL_QUEUE - 1)) * 3;
                    dst[0] = ra;
                    dst[1] = rb;
                    dst[2] = rc;
                }
                qt += n4.x + n4.y + n4.z + n4.w;
                if (qt - qh >= PL_BLOCK) {
                    group_sync();   // the queue
                    do {
                        produce(PL_BLOCK, 0);
                        qh += PL_BLOCK;
                    } while (qt - qh >= PL_BLOCK);
                }
            }
            group_sync();
            produce(qt - qh, PL_LAST);
            group_sync();   // the next item's queue starts at slot 0
        }
        if (COUNT) {
            for (int o = 16; o > 0; o >>= 1) pairs += __shfl_xor_sync(0xffffffffu, pairs, o);
            if (lane == 0 && pairs) atomicAdd(&g_plane_pairs, pairs);
        }
    } else if (warp < PL_PROD + PL_EPI) {
        // ------------------------------------------------ epilogue -------------------------------------
        // lanes of quadrant e: B' hi rows (e = 0, 1) against A hi + A lo, B' lo rows (e = 2, 3) against A hi
        const int e = warp & 3;   // the quadrant of TMEM lanes this warp may read
        int n = 0;
        for (int work = blockIdx.x; work < P.nwork; work += gridDim.x, n++) {
            const int a = n & 1;
            bool wt = true;
            if (lane == 0) {
                wt = bar_wait(tc::smem_u32(accfull + a), (uint32_t)((n >> 1) & 1), P.err);
                if (!wt) report_timeout(P.err, 5, n, a, (n >> 1) & 1, 0, 0);
            }
            if (__shfl_sync(0xffffffffu, wt ? 1 : 0, 0) == 0) break;
            tc::fence_after();
            const bool some = *reinterpret_cast<volatile int *>(have + a) != 0;
            const uint32_t base = tmem + (uint32_t)a * PL_ACC + ((uint32_t)(32 * e) << 16);
            float *dst = P.partial + (int64_t)work * 2 * ncol * 128 + 32 * e + lane;
            for (int half = 0; half < 2; half++)
                for (int c0 = 0; c0 < ncol; c0 += 8) {
                    float v[8], lo[8];
                    if (some) {
                        tc::ld8(base + (uint32_t)(128 * half + c0), v);
                        if (e < 2) tc::ld8(base + (uint32_t)(128 * half + 64 + c0), lo);
                    }
#pragma unroll
                    for (int u = 0; u < 8; u++)
                        if (c0 + u < ncol)
                            dst[(int64_t)(half * ncol + c0 + u) * 128] = some ? (e < 2 ? v[u] + lo[u] : v[u]) : 0.f;
                }
            tc::fence_before();
            __syncwarp();
            if (lane == 0) bar_arrive(tc::smem_u32(accfree + a));
        }
    } else if (lane == 0) {
        // ------------------------------------------------ MMA issuer -----------------------------------
        const uint32_t idesc = tc::instr_desc(256, 128);
        uint32_t fullpar = 0;   // bit g = parity of stage g's next full phase
        bool ok = true;
        int n = 0, taken = 0;
        for (int work = blockIdx.x; work < P.nwork && ok; work += gridDim.x, n++) {
            const int a = n & 1;
            const uint32_t acc = tmem + (uint32_t)a * PL_ACC;
            if (n >= 2 && !bar_wait(tc::smem_u32(accfree + a), (uint32_t)(((n >> 1) - 1) & 1), P.err)) {
                report_timeout(P.err, 4, taken, a, ((n >> 1) - 1) & 1, 0, taken);
                break;
            }
            tc::fence_after();
            uint32_t started = 0;
            unsigned active = (1u << PL_GROUPS) - 1u;
            for (int g = 0; active != 0u; g = (g + 1 == PL_GROUPS) ? 0 : g + 1) {
                if (!((active >> g) & 1u)) continue;
                const uint32_t par = (fullpar >> g) & 1u;
                if (!bar_wait(tc::smem_u32(full + g), par, P.err)) {
                    report_timeout(P.err, 3, taken, g, (int)par, 0, taken);
                    ok = false;
                    break;
                }
                fullpar ^= 1u << g;
                taken++;
                const int hd = *reinterpret_cast<volatile int *>(hdr + g), nb = hd & (PL_LAST - 1);
                if (hd & PL_LAST) active &= ~(1u << g);
                if (nb == 0) {
                    bar_arrive(tc::smem_u32(empty + g));
                    continue;
                }
                tc::fence_after();
                // accumulator lane m = row of [B'_hi; B'_lo], column n = row of the A copies
                const uint32_t sa = tc::smem_u32(smem + g * PL_STAGE);
#pragma unroll
                for (int ks = 0; ks < PL_GW; ks++)
                    if (ks * PL_KB < nb) {
                        tc::mma_f16(acc, tc::smem_desc_sw32(sa + ks * PL_OPS + 4 * PL_COPY),
                                    tc::smem_desc_sw32(sa + ks * PL_OPS), idesc, started);
                        started = 1u;
                    }
                tc::commit(tc::smem_u32(empty + g));
            }
            if (!ok) break;
            have[a] = started ? 1 : 0;
            bar_arrive(tc::smem_u32(accfull + a));
            tc::commit(tc::smem_u32(accfull + a));
        }
        // every MMA complete before the tensor memory is freed
        tc::commit(tc::smem_u32(done));
        if (!tc::mbar_wait(tc::smem_u32(done), 0)) tc::mbar_drain(tc::smem_u32(done), 0);
    }
    __syncwarp();
    tc::fence_before();
    __syncthreads();
    if (warp == PL_WARPS - 1) tc::dealloc(tmem, 2 * PL_ACC);
}

// u(x_i, x_j) of every sample: the items' partial sums in a fixed order, FP64.  A block takes 64 consecutive
// (column, point) outputs of one tile and sample, PL_RG groups of 64 threads striding over the items: the grid of a
// launch is small, so the loads in flight come from the groups (8.3 -> 3.2 ms per 250 samples of 456 items against
// 4 groups).
constexpr int PL_RG = 16;
__global__ void __launch_bounds__(64 * PL_RG) plane_reduce_kernel(const float *__restrict__ partial,
                                                          const int32_t *__restrict__ item_start, int first_item,
                                                          int nitems, int first_tile, int blocks_per_tile, int n0, int n1,
                                                          int T0, int T1, int nt1, const float *__restrict__ amax,
                                                          float *__restrict__ u, int64_t u_stride) {
    __shared__ double sh[PL_RG][64][2];
    const int samp = blockIdx.y, t = first_tile + blockIdx.x / blocks_per_tile;
    const int J = (T1 + 3) >> 2, I = (T0 + 3) >> 2, MI = (4 * I + 7) / 8 * 8, ncol = 12 * J;
    const int o = (blockIdx.x % blocks_per_tile) * 64 + (threadIdx.x & 63), g = threadIdx.x >> 6;
    // lane of B' (point i = h I + m at row 4 m + h) fastest, then the column (row j = h J + t, component c, at
    // 4 (3 t + c) + h)
    const int li = o % (4 * I), col = o / (4 * I);
    double re = 0.0, im = 0.0;
    if (col < ncol) {
        const int b = item_start[t] - first_item, e = item_start[t + 1] - first_item;
        for (int it = b + g; it < e; it += PL_RG) {
            const float *p = partial + (((int64_t)samp * nitems + it) * 2 * ncol + col) * 128 + li;
            const float *pi = p + (int64_t)ncol * 128;
            re += (double)((p[0] + p[64]) - (pi[MI] + pi[64 + MI]));
            im += (double)((p[MI] + p[64 + MI]) + (pi[0] + pi[64]));
        }
    }
    sh[g][threadIdx.x & 63][0] = re;
    sh[g][threadIdx.x & 63][1] = im;
    __syncthreads();
    if (g == 0 && col < ncol) {
        const int i = (li & 3) * I + (li >> 2), n = col >> 2, j = (col & 3) * J + n / 3, c = n % 3;
        const int gi = (t / nt1) * T0 + i, gj = (t % nt1) * T1 + j;
        if (i < T0 && j < T1 && gi < n0 && gj < n1) {
            const int x = threadIdx.x;
            const double inv = 1.0 / ((double)plane_scale(amax[samp]) * (double)PL_SB);
            float *dst = u + samp * u_stride + ((int64_t)gi * n1 + gj) * 6 + 2 * c;
#pragma unroll
            for (int q = 1; q < PL_RG; q++) {
                re += sh[q][x][0];
                im += sh[q][x][1];
            }
            dst[0] = (float)(re * inv);
            dst[1] = (float)(im * inv);
        }
    }
}

}  // namespace

// the plane kernel takes single-plane lattices with uniform axes 0 and 1
bool plane_tc_eligible(const LatticePlan &plan) {
    return plan.n[2] == 1 && plan.T[2] == 1 && (plan.uniform[0] || plan.n[0] == 1) &&
           (plan.uniform[1] || plan.n[1] == 1) && plan.T[0] <= PL_T0_MAX && plan.T[1] <= PL_T1_MAX;
}

void tile_shape_plane(const fga_lattice &L, int T[3]) {
    T[2] = 1;
    const int nt1 = (L.n[1] + PL_T1_MAX - 1) / PL_T1_MAX;
    T[1] = (L.n[1] + nt1 - 1) / nt1;
    const int nt0 = (L.n[0] + PL_T0_MAX - 1) / PL_T0_MAX;
    T[0] = (L.n[0] + nt0 - 1) / nt0;
}

fga_status run_plane_tc(Workspace &ws, const LatticePlan &plan, const void *rec, int64_t rec_stride, int ns, double k,
                        double rw, void *u, int64_t u_stride, cudaStream_t s, int cat, const float *amax_in) {
    const int T0 = plan.T[0], T1 = plan.T[1], ncol = 12 * ((T1 + 3) / 4);
    const size_t per_item = sizeof(float) * 2 * (size_t)ncol * 128;
    // partial sums of at most PLANE_PARTIAL_MAX bytes per launch: as many samples as fit, or else as many tiles (the
    // same where that much does not fit the device or the caller's bound)
    const size_t max_items = PLANE_PARTIAL_MAX / per_item;
    const int32_t *starts = plan.h_item_start;
    int tile_items = 1;   // items of the largest tile
    for (int t = 0; t < plan.ntiles; t++) tile_items = std::max(tile_items, starts[t + 1] - starts[t]);
    int chunk = (int)std::max<size_t>(1, std::min<size_t>({(size_t)ns, max_items / std::max(plan.nitems, 1), 65535}));
    int most = std::max(plan.nitems, 1);   // items of a launch and sample
    if ((size_t)plan.nitems > max_items) most = std::max((int)max_items, tile_items);
    auto bytes = [&](int items, int samples) { return per_item * (size_t)items * (size_t)samples; };
    fga_status fits = ensure_scratch(ws.partial, chunk, 1, [&](int c) { return bytes(most, c) + 64; });
    if (fits == FGA_ERR_OOM) fits = ensure_scratch(ws.partial, most, tile_items, [&](int m) { return bytes(m, 1) + 64; });
    FGA_TRY(fits);
    const bool by_tile = plan.nitems > most;
    const size_t pbytes = bytes(most, chunk);
    float *amax = reinterpret_cast<float *>(ws.partial.as<char>() + pbytes);
    if (!ws.status.p) FGA_TRY(status_reset(ws, s));
    prof_add_pairs_tested(plan.pairs_tested * ns);
    if (!amax_in) {   // one sample
        FGA_CUDA(cudaMemsetAsync(amax, 0, 64, s));
        if (plan.nitems > 0) FGA_TRY(rec_absmax(static_cast<const float *>(rec), plan.n_rec, amax, s, cat));
    }
    int dev = 0, sms = 152;
    FGA_CUDA(cudaGetDevice(&dev));
    FGA_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    const int J = (T1 + 3) / 4, I = (T0 + 3) / 4;
    const bool cnt = prof_counting();
    for (int s0 = 0; s0 < ns; s0 += chunk)
        for (int t0 = 0; t0 < plan.ntiles;) {
            const int m = std::min(chunk, ns - s0);
            int t1 = plan.ntiles, i0 = 0, i1 = plan.nitems;
            if (by_tile) {
                i0 = starts[t0];
                t1 = t0 + 1;
                while (t1 < plan.ntiles && starts[t1 + 1] - i0 <= most) t1++;
                i1 = starts[t1];
            }
            const float *am = amax_in ? amax_in + s0 : amax;
            if (i1 > i0) {
                PlaneArgs A;
                A.rec = static_cast<const float *>(rec) + rec_stride * s0;
                A.rec_stride = rec_stride;
                A.items = plan.items + i0;
                A.nitems = i1 - i0;
                A.nwork = A.nitems * m;
                A.n0 = plan.n[0];
                A.n1 = plan.n[1];
                A.T0 = T0;
                A.T1 = T1;
                A.nt1 = plan.nt[1];
                A.x0 = (float)plan.x_first[0];
                A.h0 = (float)plan.dx[0];
                A.x1 = (float)plan.x_first[1];
                A.h1 = (float)plan.dx[1];
                A.x2 = (float)plan.x_first[2];
                A.k = (float)k;
                A.rw2 = (float)(rw * rw);
                A.amax = am;
                A.partial = ws.partial.as<float>();
                A.err = ws.status.as<int>();
                const int grid = std::min(A.nwork, sms);
                ProfScope ps(cat, s);
#define FGA_PLANE(CNT, JT, IT)                                                                                    \
        do {                                                                                                          \
            FGA_CUDA(cudaFuncSetAttribute(plane_tc_kernel<CNT, JT, IT>, cudaFuncAttributeMaxDynamicSharedMemorySize,  \
                                          PL_SMEM));                                                                  \
            plane_tc_kernel<CNT, JT, IT><<<grid, PL_THREADS, PL_SMEM, s>>>(A);                                        \
        } while (0)
                // Tiles of 17 to 20 and of 13 to 16 points on both axes (quarters of 5 x 5 and 4 x 4 points) have their loops
                // unrolled, which takes a seventh off the sums: 138.6 -> 117.7 ms on 250 samples of 8.4 M beams on 20 x 20
                // receivers, 31.4 -> 26.9 ms on 200 of 2.7 M on 16 x 16.  Other tiles take the general loops: a variant for each
                // of the 30 pairs of quarters would multiply the build.
                if (cnt) FGA_PLANE(true, 0, 0);
                else if (J == 5 && I == 5) FGA_PLANE(false, 5, 5);
                else if (J == 4 && I == 4) FGA_PLANE(false, 4, 4);
                else FGA_PLANE(false, 0, 0);
#undef FGA_PLANE
                FGA_CUDA(cudaGetLastError());
            }
            ProfScope ps(P_REDUCE, s);
            const int per_tile = (ncol * 4 * I + 63) / 64;
            const dim3 rgrid((unsigned)per_tile * (unsigned)(t1 - t0), (unsigned)m);
            plane_reduce_kernel<<<rgrid, 64 * PL_RG, 0, s>>>(ws.partial.as<float>(), plan.item_start, i0, i1 - i0, t0, per_tile,
                                                      plan.n[0], plan.n[1], T0, T1, plan.nt[1], am,
                                                      static_cast<float *>(u) + u_stride * s0, u_stride);
            FGA_CUDA(cudaGetLastError());
            t0 = t1;
        }
    return FGA_OK;
}

}  // namespace fga
