// Complex GEMMs of the wave-packet transform (A1) on the 5th-generation tensor cores, FP16 split
// precision with FP32 accumulation:
//
//   C[z][m][n] = scale * sum_k A[z][m][k] B[n][k]        (complex; B = a per-axis kernel matrix, |B| <= 1)
//
// Complex -> real: with B' = [Re B ; Im B] (rows n: Re, rows n_c + n: Im), D_re = Re A B'^T and D_im = Im A B'^T go
// to two accumulators and Re C = D_re[n] - D_im[n_c + n], Im C = D_re[n_c + n] + D_im[n] are formed when they are
// read back.  FP16 split: x = hi + lo with hi = fp16(x), lo = fp16(x - hi); each real product is hi*hi + hi*lo + lo*hi
// (the lo*lo term is below FP32 rounding), three tcgen05.mma per K step.  Operands are scaled by exact powers of two
// so that hi and lo stay in the FP16 normal range (A by a bound on |A| read from device memory, B by 2^14).
//
// B is evaluated once per transform, already split and in the operand layout (kernel_matrix_kernel), so that a K
// block of it is one bulk copy; converting it again in every CTA cost more than converting A.
//
// One CTA = one 128-row M tile x one N tile (n_c <= 64), 256 threads, two CTAs per SM: every thread loads its part of
// the next K block of A into registers (2 x 8 complex values) while the tensor cores work, splits it into one of two
// shared-memory stages in the canonical no-swizzle K-major layout (8x8 core matrices of 128 contiguous bytes; a quarter
// warp's 16-byte stores fill one), one elected thread issues the MMAs and commits them to the stage's mbarrier.
// Bound by the HBM stream of its operands and results and by the conversions.  Bench transform (128^3 x 3 to
// 192^3 x 3): the three stages 1,020 -> 336 us (single-buffered CTAs of 128 threads that converted both operands in every
// CTA and read the components in three passes), the whole call 1.17 -> 0.46 ms.
// Every wait is bounded: a wait that runs out sets *err, waits once more (bounded) for the outstanding commits, and
// then frees its tensor memory without writing C.
#include <cuda_fp16.h>

#include <algorithm>
#include <cmath>

#include "fga_beam.cuh"
#include "tc_gemm.cuh"
#include "tcgen05.cuh"

namespace fga {
namespace {

constexpr int TC_M = 128;      // rows per tile (TMEM lanes)
constexpr int TC_THREADS = 256;
constexpr int TC_A_BYTES = TC_M * TC_KB * 2;           // one copy of a K block of A': 8 KB
constexpr int TC_B_BYTES = 2 * TC_NC * TC_KB * 2;      // one copy of a K block of B' (n_c = TC_NC): 8 KB
constexpr int TC_STAGE = 4 * TC_A_BYTES + 2 * TC_B_BYTES;   // Re hi, Re lo, Im hi, Im lo of A; hi, lo of B'
constexpr int TC_SMEM = 2 * TC_STAGE + 128 + 1024;
constexpr uint32_t TC_TMEM_COLS = 256;

template <typename TA> struct GemmArgs {
    const TA *A;
    const unsigned char *B;   // split kernel matrix: [N tile][K block][hi, lo][2 nc rows][TC_KB]
    float2 *C;
    int64_t sAz, sAm, sAk, sCz, sCm, sCn;   // row m at (m / rdiv) s?m + m % rdiv
    int rdiv;
    int64_t M;
    int N, K, nc, ntile, nkb;
    float scale;
    const float *amax;
    float amax_factor;
    int *err;
};

// grid: (M tiles x N tiles, Z), the N tiles of an M tile next to each other (they share A in L2)
template <typename TA> __global__ void __launch_bounds__(TC_THREADS, 2) tc_cgemm_kernel(GemmArgs<TA> G) {
    extern __shared__ unsigned char smem_raw[];
    unsigned char *smem = smem_raw + ((1024 - (tc::smem_u32(smem_raw) & 1023)) & 1023);
    uint64_t *mma_done = reinterpret_cast<uint64_t *>(smem + 2 * TC_STAGE);   // [2] the stage's MMAs are complete
    uint64_t *b_full = mma_done + 2;                                          // [2] the stage's B block has arrived
    uint64_t *fin = b_full + 2;                                               // give-up path
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(fin + 1);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int z = blockIdx.y, nt = blockIdx.x % G.ntile;
    const int64_t m0 = (int64_t)(blockIdx.x / G.ntile) * TC_M;
    const int n0 = nt * G.nc;
    const int nc = min(G.nc, G.N - n0);   // complex columns of this tile
    const uint32_t NR = 2 * G.nc;         // real MMA width (unused rows of B' are zero)
    const uint32_t bbytes = NR * TC_KB * 2;

    // operand scales: A so that |A| * sa <= 2^14, B (|B| <= 1) by 2^14
    float sa = 1.0f;
    {
        const float bound = (*G.amax) * G.amax_factor;
        if (bound > 0.0f && isfinite(bound)) {
            int e;
            frexpf(bound, &e);          // bound < 2^e
            sa = ldexpf(1.0f, 14 - e);
        }
    }
    if (warp == 0) tc::alloc(tc::smem_u32(tmem_slot), TC_TMEM_COLS);
    if (tid == 0) {
        for (int s = 0; s < 2; s++) {
            tc::mbar_init(tc::smem_u32(mma_done + s));
            tc::mbar_init(tc::smem_u32(b_full + s));
        }
        tc::mbar_init(tc::smem_u32(fin));
    }
    tc::fence_before();
    __syncthreads();
    tc::fence_after();
    const uint32_t tmem = *tmem_slot;
    const uint32_t idesc = tc::instr_desc((int)NR, TC_M);

    // this thread's two tasks of a K block: row tid & 127, 8 consecutive k from 8 ((tid >> 7) + 2 j)
    const int row = tid & 127, kq = tid >> 7;
    const int64_t gm = m0 + row;
    const bool rok = gm < G.M;
    const TA *arow = G.A + (int64_t)z * G.sAz + (rok ? (gm / G.rdiv) * G.sAm + gm % G.rdiv : 0);
    float2 v[2][8];
    auto load = [&](int kb) {
#pragma unroll
        for (int j = 0; j < 2; j++)
#pragma unroll
            for (int u = 0; u < 8; u++) {
                const int k = kb * TC_KB + 8 * (kq + 2 * j) + u;
                v[j][u] = rok && k < G.K ? tc::ld_c<TA>(arow + (int64_t)k * G.sAk) : make_float2(0.f, 0.f);
            }
    };
    load(0);
    bool ok = true;
    int stuck = -1;   // block whose copy of B was not seen to arrive
    for (int kb = 0; kb < G.nkb && ok; kb++) {
        unsigned char *st = smem + (kb & 1) * TC_STAGE;
        // the MMAs that read this stage two blocks ago
        bool arrived = true;
        if (kb >= 2 && tid == 0) arrived = tc::mbar_wait(tc::smem_u32(mma_done + (kb & 1)), (uint32_t)(((kb >> 1) - 1) & 1));
        if (kb >= 2) ok = __syncthreads_and(arrived ? 1 : 0) != 0;   // uniform across the CTA
        if (!ok) break;
        if (tid == 0) {
            const uint32_t bar = tc::smem_u32(b_full + (kb & 1));
            const unsigned char *src = G.B + ((int64_t)nt * G.nkb + kb) * 2 * bbytes;
            asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(2 * bbytes) : "memory");
            asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                             tc::smem_u32(st + 4 * TC_A_BYTES)),
                         "l"(src), "r"(2 * bbytes), "r"(bar)
                         : "memory");
        }
#pragma unroll
        for (int j = 0; j < 2; j++) {
            float re[8], im[8];
#pragma unroll
            for (int u = 0; u < 8; u++) {
                re[u] = v[j][u].x;
                im[u] = v[j][u].y;
            }
            const uint32_t off = tc::kmaj_off(row, 8 * (kq + 2 * j));
            tc::split8(st, st + TC_A_BYTES, off, re, sa);
            tc::split8(st + 2 * TC_A_BYTES, st + 3 * TC_A_BYTES, off, im, sa);
        }
        if (kb + 1 < G.nkb) load(kb + 1);
        // make the generic-proxy stores visible to the tensor cores, then issue
        tc::fence_async_smem();
        tc::fence_before();
        __syncthreads();
        tc::fence_after();
        if (tid == 0) {
            arrived = tc::mbar_wait(tc::smem_u32(b_full + (kb & 1)), (uint32_t)((kb >> 1) & 1));
            if (arrived) {
                const uint32_t a0 = tc::smem_u32(st), b0 = a0 + 4 * TC_A_BYTES;
#pragma unroll
                for (int half = 0; half < 2; half++)   // Re A, Im A
#pragma unroll
                    for (int ks = 0; ks < TC_KB / 16; ks++) {
                        const uint32_t ko = ks * 2 * 128;   // two core matrices along K
                        const uint64_t ah = tc::smem_desc(a0 + (2 * half) * TC_A_BYTES + ko),
                                       al = tc::smem_desc(a0 + (2 * half + 1) * TC_A_BYTES + ko);
                        const uint64_t bh = tc::smem_desc(b0 + ko), bl = tc::smem_desc(b0 + bbytes + ko);
                        const uint32_t d = tmem + (uint32_t)half * NR;
                        tc::mma_f16(d, ah, bh, idesc, kb > 0 || ks > 0 ? 1u : 0u);
                        tc::mma_f16(d, ah, bl, idesc, 1u);
                        tc::mma_f16(d, al, bh, idesc, 1u);
                    }
                tc::commit(tc::smem_u32(mma_done + (kb & 1)));
            }
        }
        ok = __syncthreads_and(tid != 0 || arrived ? 1 : 0) != 0;   // a B block that never came: every thread stops
        if (!ok) stuck = kb;
    }
    // the last one or two blocks' MMAs
    if (ok) {
        bool arrived = true;
        if (tid == 0)
            for (int kb = max(0, G.nkb - 2); kb < G.nkb; kb++)
                arrived = tc::mbar_wait(tc::smem_u32(mma_done + (kb & 1)), (uint32_t)((kb >> 1) & 1)) && arrived;
        ok = __syncthreads_and(arrived ? 1 : 0) != 0;
        tc::fence_after();
    }
    // give-up: report, and let the outstanding MMAs and the copy of block `stuck` land before freeing the columns
    if (!ok && tid == 0) {
        atomicExch(G.err, 1);
        tc::commit(tc::smem_u32(fin));
        tc::mbar_drain(tc::smem_u32(fin), 0);
        if (stuck >= 0) tc::mbar_drain(tc::smem_u32(b_full + (stuck & 1)), (uint32_t)((stuck >> 1) & 1));
    }
    if (ok) {
        // ---- epilogue: warp w owns TMEM lanes (rows) 32 (w % 4) .. + 31 and the 8-column chunks w / 4, + 2, ... ----
        const int64_t m = m0 + (warp & 3) * 32 + lane;
        const float inv = G.scale / (sa * TC_SB);
        const uint32_t base = tmem + ((uint32_t)((warp & 3) * 32) << 16);
        float2 *crow = G.C + (int64_t)z * G.sCz + (m < G.M ? (m / G.rdiv) * G.sCm + m % G.rdiv : 0);
        for (int c0 = (warp >> 2) * 8; c0 < nc; c0 += 16) {
            float rr[8], ri[8], ir[8], ii[8];
            tc::ld8(base + (uint32_t)c0, rr);
            tc::ld8(base + (uint32_t)(G.nc + c0), ri);
            tc::ld8(base + NR + (uint32_t)c0, ir);
            tc::ld8(base + NR + (uint32_t)(G.nc + c0), ii);
            if (m < G.M)
#pragma unroll
                for (int q = 0; q < 8; q++)
                    if (c0 + q < nc)
                        crow[(int64_t)(n0 + c0 + q) * G.sCn] = make_float2((rr[q] - ii[q]) * inv, (ri[q] + ir[q]) * inv);
        }
    }
    tc::fence_before();
    __syncthreads();
    if (warp == 0) tc::dealloc(tmem, TC_TMEM_COLS);
}

// K[a][i] = exp(-i k p (y_i - q) - k (y_i - q)^2 / 2), a = iq np + jp, of the three axes (blockIdx.y), scaled by 2^14
// and split to FP16 hi and lo in the layout a K block is copied in: [N tile][K block][hi, lo][rows Re 0 .. n_c-1, Im
// n_c .. 2 n_c-1][TC_KB], zero beyond the matrix
__global__ void kernel_matrix_kernel(KernelMatrices P) {
    const int ax = blockIdx.y;
    const KernelMatrix &X = P.ax[ax];
    const int kpad = X.nkb * TC_KB, idx = blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= X.ntile * X.nc * kpad) return;
    const int a = idx / kpad, i = idx % kpad;   // padded row and column
    float re = 0.f, im = 0.f;
    if (a < P.nq * P.np && i < X.ny) {
        const int iq = a / P.np, jp = a % P.np;
        const double q = X.q0 + iq * X.dq, p = X.p0 + jp * X.dp, y = X.y0 + i * X.dy;
        const double d = y - q;
        double s, c;
        sincos(-P.k * p * d, &s, &c);
        const double e = exp(-0.5 * P.k * d * d);
        re = (float)(e * c) * TC_SB;
        im = (float)(e * s) * TC_SB;
    }
    const int t = a / X.nc, j = a % X.nc, kb = i / TC_KB, kk = i % TC_KB;
    const int64_t copy = (int64_t)2 * X.nc * TC_KB * 2;   // bytes of one copy
    unsigned char *blk = X.B + ((int64_t)t * X.nkb + kb) * 2 * copy;
    tc::split_store(blk, blk + copy, tc::kmaj_off(j, kk), re);
    tc::split_store(blk, blk + copy, tc::kmaj_off(X.nc + j, kk), im);
}

// largest |Re|, |Im|: compared as integers (bits of non-negative doubles order like their values; NaN is passed over),
// four values in flight per thread
__global__ void __launch_bounds__(256) absmax_kernel(const double2 *__restrict__ x, int64_t n, float *__restrict__ out) {
    const long long inf = 0x7ff0000000000000ll;
    long long m = 0;
    auto take = [&](double v) {
        const long long b = __double_as_longlong(v) & 0x7fffffffffffffffll;
        if (b > m && b <= inf) m = b;
    };
    const int64_t step = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += 4 * step) {
        double2 v[4];
#pragma unroll
        for (int u = 0; u < 4; u++) v[u] = i + u * step < n ? x[i + u * step] : make_double2(0.0, 0.0);
#pragma unroll
        for (int u = 0; u < 4; u++) {
            take(v[u].x);
            take(v[u].y);
        }
    }
    float f = (float)__longlong_as_double(m);
    for (int o = 16; o > 0; o >>= 1) f = fmaxf(f, __shfl_xor_sync(0xffffffffu, f, o));
    if ((threadIdx.x & 31) == 0) atomicMax(reinterpret_cast<int *>(out), __float_as_int(f));  // f >= 0
}

}  // namespace

// |x|_max of complex double data into *out (DEVICE float, zeroed here)
fga_status tc_absmax(const double2 *x, int64_t n, float *out, cudaStream_t s) {
    FGA_CUDA(cudaMemsetAsync(out, 0, sizeof(float), s));
    const int blocks = (int)std::min<int64_t>(152 * 8, (n + 255) / 256 + 1);
    absmax_kernel<<<blocks, 256, 0, s>>>(x, n, out);
    FGA_CUDA(cudaGetLastError());
    return FGA_OK;
}

void tc_kernel_shape(int N, int K, KernelMatrix &X) {
    X.ny = K;
    X.ntile = (N + TC_NC - 1) / TC_NC;
    X.nc = ((N + X.ntile - 1) / X.ntile + 7) / 8 * 8;
    X.nkb = (K + TC_KB - 1) / TC_KB;
    X.bytes = (size_t)X.ntile * X.nkb * 2 * 2 * X.nc * TC_KB * 2;
}

fga_status tc_kernel_matrices(const KernelMatrices &P, cudaStream_t s) {
    int64_t most = 0;
    for (int a = 0; a < 3; a++) most = std::max(most, (int64_t)P.ax[a].ntile * P.ax[a].nc * P.ax[a].nkb * TC_KB);
    FGA_CHECK(most < (int64_t)1 << 31, "wave-packet transform: kernel matrix too large");
    ProfScope ps(P_DECOMP, s);
    kernel_matrix_kernel<<<dim3((unsigned)((most + 255) / 256), 3), 256, 0, s>>>(P);
    FGA_CUDA(cudaGetLastError());
    return FGA_OK;
}

template <typename TA>
fga_status tc_cgemm(const TA *A, int64_t sAz, int64_t sAm, int64_t sAk, const KernelMatrix &X, float2 *C, int64_t sCz,
                    int64_t sCm, int64_t sCn, int rdiv, int Z, int64_t M, int N, float scale, const float *amax,
                    float amax_factor, int *err, cudaStream_t s) {
    GemmArgs<TA> G{A, X.B, C, sAz, sAm, sAk, sCz, sCm, sCn, rdiv, M, N, X.ny, X.nc, X.ntile, X.nkb, scale, amax, amax_factor, err};
    FGA_CUDA(cudaFuncSetAttribute(tc_cgemm_kernel<TA>, cudaFuncAttributeMaxDynamicSharedMemorySize, TC_SMEM));
    // at most 65,535 batches per launch
    for (int z0 = 0; z0 < Z; z0 += 65535) {
        const dim3 grid((unsigned)((M + TC_M - 1) / TC_M) * (unsigned)X.ntile, (unsigned)std::min(65535, Z - z0));
        ProfScope ps(P_DECOMP, s);
        tc_cgemm_kernel<TA><<<grid, TC_THREADS, TC_SMEM, s>>>(G);
        FGA_CUDA(cudaGetLastError());
        G.A += (int64_t)65535 * sAz;
        G.C += (int64_t)65535 * sCz;
    }
    return FGA_OK;
}

template fga_status tc_cgemm<double2>(const double2 *, int64_t, int64_t, int64_t, const KernelMatrix &, float2 *, int64_t,
                                      int64_t, int64_t, int, int, int64_t, int, float, const float *, float, int *,
                                      cudaStream_t);
template fga_status tc_cgemm<float2>(const float2 *, int64_t, int64_t, int64_t, const KernelMatrix &, float2 *, int64_t,
                                     int64_t, int64_t, int, int, int64_t, int, float, const float *, float, int *,
                                     cudaStream_t);

}  // namespace fga
