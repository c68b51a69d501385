// A5-A6: cell binning of beam centres (stable LSD radix sort) and the truncated Gaussian sum of
// Eq. FGA as a gather: every CTA owns one tile of up to 32 points of one cell and one chunk of the
// beams sitting in that cell's 27 neighbours; partial sums go to scratch and a second kernel adds
// them in a fixed order (no atomics, deterministic).
#include <algorithm>
#include <cmath>
#include <cstddef>
#include <cstring>
#include <numeric>

#include "fga_beam.cuh"
#include "gather.cuh"

namespace fga {

// ---------------------------------------------------------------------------------------------
// keys
// ---------------------------------------------------------------------------------------------
// The sort's tile: RS_T threads of RS_I items each (16 items halve the counts to scan, but the scatter's rounds are
// serial: 9 -> 17 us at 0.9 M centres).
constexpr int RS_T = 256, RS_I = 8, RS_TILE = RS_T * RS_I;

// Bucket of every centre (-1: not sorted, with drop the centres outside an unclamped grid and dead beams) and the tile's
// counts of the first digit.
template <typename TQ>
__global__ void __launch_bounds__(RS_T) keys_kernel(BinGrid g, const TQ *__restrict__ Q, int64_t sb, int64_t sd, int64_t n,
                                                   const int32_t *__restrict__ cls, bool drop, int32_t *__restrict__ keys,
                                                   int digits, int ntiles, uint32_t *__restrict__ hist) {
    __shared__ uint32_t cnt[256];
    cnt[threadIdx.x] = 0;
    __syncthreads();
#pragma unroll 2
    for (int r = 0; r < RS_I; r++) {
        const int64_t b = (int64_t)blockIdx.x * RS_TILE + r * RS_T + threadIdx.x;
        if (b >= n) break;
        int cell[3];
        bool inside = true;
#pragma unroll
        for (int d = 0; d < 3; d++) {
            const float q = (float)Q[b * sb + d * sd];
            const float t = __fmul_rn(__fsub_rn(q, g.o[d]), g.inv_h);
            const float fl = floorf(t);
            int cd;
            if (!(fl >= 0.0f)) {
                cd = 0;
                inside = false;
            } else if (fl > (float)(g.nc[d] - 1)) {
                cd = g.nc[d] - 1;
                inside = false;
            } else {
                cd = (int)fl;
            }
            cell[d] = cd;
        }
        int key = (cell[0] * g.nc[1] + cell[1]) * g.nc[2] + cell[2];
        const bool out = !g.clamp && (!inside || (cls && (cls[b] & FL_DEAD)));
        if (out) key = g.ncells;
        if (cls) key += (cls[b] & FL_CLASS_MASK) * (g.ncells + 1);
        if (out && drop) key = -1;
        keys[b] = key;
        if (key >= 0) atomicAdd(&cnt[key & (digits - 1)], 1u);
    }
    __syncthreads();
    if ((int)threadIdx.x < digits) hist[(int64_t)threadIdx.x * ntiles + blockIdx.x] = cnt[threadIdx.x];
    if (blockIdx.x == 0 && threadIdx.x == 0) hist[(int64_t)digits * ntiles] = 0;   // the scan leaves the total here
}

// ---------------------------------------------------------------------------------------------
// stable LSD radix sort of (key, index) pairs, digits of up to 8 bits; the number of pairs is on the device (cnt) from
// the second pass on
// ---------------------------------------------------------------------------------------------
__global__ void __launch_bounds__(RS_T) rs_hist_kernel(const int32_t *__restrict__ keys, const uint32_t *__restrict__ count,
                                                      int shift, int digits, int ntiles, uint32_t *__restrict__ hist) {
    __shared__ uint32_t cnt[256];
    cnt[threadIdx.x] = 0;
    __syncthreads();
    const int64_t base = (int64_t)blockIdx.x * RS_TILE, n = *count;
#pragma unroll 8
    for (int r = 0; r < RS_I; r++) {
        const int64_t i = base + r * RS_T + threadIdx.x;
        if (i < n) atomicAdd(&cnt[(keys[i] >> shift) & (digits - 1)], 1u);
    }
    __syncthreads();
    if ((int)threadIdx.x < digits) hist[(int64_t)threadIdx.x * ntiles + blockIdx.x] = cnt[threadIdx.x];
    if (blockIdx.x == 0 && threadIdx.x == 0) hist[(int64_t)digits * ntiles] = 0;
}

// vin NULL: the first pass, whose values are the indexes and whose keys may be -1; it leaves the total in *count
__global__ void __launch_bounds__(RS_T) rs_scatter_kernel(const int32_t *__restrict__ kin, const int32_t *__restrict__ vin,
                                                         int64_t n, uint32_t *__restrict__ count, int shift, int digits,
                                                         int ntiles, const uint32_t *__restrict__ off,
                                                         int32_t *__restrict__ kout, int32_t *__restrict__ vout) {
    __shared__ uint32_t run[256];
    __shared__ uint32_t wcnt[RS_T / 32][256];
    __shared__ uint32_t woff[RS_T / 32][256];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int64_t base = (int64_t)blockIdx.x * RS_TILE;
    if (vin) {
        n = *count;
        if (base >= n) return;
    } else if (blockIdx.x == 0 && tid == 0) {
        *count = off[(int64_t)digits * ntiles];
    }
    run[tid] = 0;
#pragma unroll
    for (int w = 0; w < RS_T / 32; w++) wcnt[w][tid] = 0;
    __syncthreads();
    const unsigned lt = (1u << lane) - 1u;
    for (int r = 0; r < RS_I; r++) {
        const int64_t i = base + r * RS_T + tid;
        const int32_t key = i < n ? kin[i] : -1;
        const bool valid = key >= 0;
        const int32_t val = valid && vin ? vin[i] : (int32_t)i;
        const int digit = valid ? ((key >> shift) & (digits - 1)) : 256;
        const unsigned peers = __match_any_sync(0xffffffffu, digit);
        const int rank = __popc(peers & lt);
        if (valid && (__ffs(peers) - 1) == lane) wcnt[warp][digit] = __popc(peers);
        __syncthreads();
        {
            uint32_t acc = run[tid];
#pragma unroll
            for (int w = 0; w < RS_T / 32; w++) {
                const uint32_t c = wcnt[w][tid];
                woff[w][tid] = acc;
                acc += c;
                wcnt[w][tid] = 0;
            }
            run[tid] = acc;
        }
        __syncthreads();
        if (valid) {
            const uint32_t pos = off[(int64_t)digit * ntiles + blockIdx.x] + woff[warp][digit] + rank;
            kout[pos] = key;
            vout[pos] = val;
        }
    }
}

// exclusive scan in place of up to SCAN_ONE uint32 by one block, a thread's 32 all in flight at once (the three launches
// of the scan below are three gaps for a few microseconds of work)
constexpr int SCAN_ONE = 32768;
__global__ void __launch_bounds__(1024) scan_one_kernel(uint32_t *__restrict__ a, int n) {
    __shared__ uint32_t ws[32];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int per = ((n + 1023) / 1024 + 3) / 4, i0 = 4 * per * (int)threadIdx.x;   // per: groups of four
    uint4 v[8];
    uint32_t tot = 0;
#pragma unroll
    for (int j = 0; j < 8; j++) {
        const int i = i0 + 4 * j;
        v[j] = make_uint4(0, 0, 0, 0);
        if (j < per) {
            if (i + 3 < n) {
                v[j] = *reinterpret_cast<const uint4 *>(a + i);
            } else {
                if (i < n) v[j].x = a[i];
                if (i + 1 < n) v[j].y = a[i + 1];
                if (i + 2 < n) v[j].z = a[i + 2];
            }
        }
        tot += v[j].x + v[j].y + v[j].z + v[j].w;
    }
    uint32_t x = tot;
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t t = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += t;
    }
    if (lane == 31) ws[warp] = x;
    __syncthreads();
    if (warp == 0) {
        uint32_t y = ws[lane];
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t t = __shfl_up_sync(0xffffffffu, y, o);
            if (lane >= o) y += t;
        }
        ws[lane] = y;
    }
    __syncthreads();
    uint32_t run = (warp ? ws[warp - 1] : 0u) + x - tot;
#pragma unroll
    for (int j = 0; j < 8; j++) {
        const int i = i0 + 4 * j;
        const uint4 e = make_uint4(run, run + v[j].x, run + v[j].x + v[j].y, run + v[j].x + v[j].y + v[j].z);
        run = e.w + v[j].w;
        if (j < per) {
            if (i + 3 < n) {
                *reinterpret_cast<uint4 *>(a + i) = e;
            } else {
                if (i < n) a[i] = e.x;
                if (i + 1 < n) a[i + 1] = e.y;
                if (i + 2 < n) a[i + 2] = e.z;
            }
        }
    }
}

// exclusive scan of n uint32 in place: per-block scans, a one-block scan of block sums, fix-up
constexpr int SC_T = 256, SC_I = 8, SC_TILE = SC_T * SC_I;

__global__ void __launch_bounds__(SC_T) scan_block_kernel(uint32_t *__restrict__ a, int64_t n, uint32_t *__restrict__ bsum) {
    __shared__ uint32_t sh[SC_T];
    const int64_t base = (int64_t)blockIdx.x * SC_TILE + (int64_t)threadIdx.x * SC_I;
    uint32_t v[SC_I], tot = 0;
#pragma unroll
    for (int j = 0; j < SC_I; j++) {
        v[j] = (base + j < n) ? a[base + j] : 0u;
        tot += v[j];
    }
    sh[threadIdx.x] = tot;
    __syncthreads();
    for (int o = 1; o < SC_T; o <<= 1) {
        const uint32_t t = threadIdx.x >= o ? sh[threadIdx.x - o] : 0u;
        __syncthreads();
        sh[threadIdx.x] += t;
        __syncthreads();
    }
    uint32_t run = sh[threadIdx.x] - tot;  // exclusive prefix of this thread
#pragma unroll
    for (int j = 0; j < SC_I; j++) {
        if (base + j < n) a[base + j] = run;
        run += v[j];
    }
    if (threadIdx.x == SC_T - 1) bsum[blockIdx.x] = sh[SC_T - 1];
}

__global__ void __launch_bounds__(1024) scan_sums_kernel(uint32_t *__restrict__ bsum, int nb) {
    // one block; nb <= 1024 * 16
    __shared__ uint32_t sh[1024];
    const int per = (nb + 1023) / 1024;
    const int beg = threadIdx.x * per;
    uint32_t tot = 0;
    for (int j = 0; j < per; j++)
        if (beg + j < nb) tot += bsum[beg + j];
    sh[threadIdx.x] = tot;
    __syncthreads();
    for (int o = 1; o < 1024; o <<= 1) {
        const uint32_t t = threadIdx.x >= o ? sh[threadIdx.x - o] : 0u;
        __syncthreads();
        sh[threadIdx.x] += t;
        __syncthreads();
    }
    uint32_t run = sh[threadIdx.x] - tot;
    for (int j = 0; j < per; j++)
        if (beg + j < nb) {
            const uint32_t v = bsum[beg + j];
            bsum[beg + j] = run;
            run += v;
        }
}

__global__ void scan_add_kernel(uint32_t *__restrict__ a, int64_t n, const uint32_t *__restrict__ bsum) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) a[i] += bsum[i / SC_TILE];
}

fga_status scan_exclusive_u32(uint32_t *a, int64_t n, cudaStream_t s);

static fga_status exclusive_scan(Workspace &ws, uint32_t *a, int64_t n, cudaStream_t s) {
    if (n <= SCAN_ONE) {
        ProfScope ps(P_BIN, s);
        scan_one_kernel<<<1, 1024, 0, s>>>(a, (int)n);
        FGA_CUDA(cudaGetLastError());
        return FGA_OK;
    }
    const int64_t nb = (n + SC_TILE - 1) / SC_TILE;
    // more than 1024 x 16 block sums: the multi-level scan (it allocates its block sums)
    if (nb > 1024 * 16) return scan_exclusive_u32(a, n, s);
    FGA_TRY(ws.scan_blocks.ensure(sizeof(uint32_t) * (size_t)std::max<int64_t>(nb, 1)));
    uint32_t *bs = ws.scan_blocks.as<uint32_t>();
    {
        ProfScope ps(P_BIN, s);
        scan_block_kernel<<<(unsigned)nb, SC_T, 0, s>>>(a, n, bs);
    }
    {
        ProfScope ps(P_BIN, s);
        scan_sums_kernel<<<1, 1024, 0, s>>>(bs, (int)nb);
    }
    {
        ProfScope ps(P_BIN, s);
        scan_add_kernel<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(a, n, bs);
    }
    FGA_CUDA(cudaGetLastError());
    return FGA_OK;
}

// the same scan for any n < 2^32 elements: the block sums of one level are scanned by the next level
fga_status scan_exclusive_u32(uint32_t *a, int64_t n, cudaStream_t s) {
    if (n <= 0) return FGA_OK;
    const int64_t nb = (n + SC_TILE - 1) / SC_TILE;
    ScopedDevBuf sums;
    FGA_TRY(sums.ensure(sizeof(uint32_t) * (size_t)nb));
    uint32_t *bs = sums.as<uint32_t>();
    {
        ProfScope ps(P_DECOMP, s);
        scan_block_kernel<<<(unsigned)nb, SC_T, 0, s>>>(a, n, bs);
    }
    FGA_CUDA(cudaGetLastError());
    if (nb <= 1024 * 16) {
        ProfScope ps(P_DECOMP, s);
        scan_sums_kernel<<<1, 1024, 0, s>>>(bs, (int)nb);
        FGA_CUDA(cudaGetLastError());
    } else {
        FGA_TRY(scan_exclusive_u32(bs, nb, s));
    }
    {
        ProfScope ps(P_DECOMP, s);
        scan_add_kernel<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(a, n, bs);
    }
    FGA_CUDA(cudaGetLastError());
    // the block sums are released when this scope ends
    FGA_CUDA(cudaStreamSynchronize(s));
    return FGA_OK;
}

__global__ void cell_start_kernel(const int32_t *__restrict__ keys, const uint32_t *__restrict__ count, int64_t most,
                                  int nbuckets, int32_t *__restrict__ start) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x, n = count ? (int64_t)*count : 0;
    if (i > n || i > most) return;
    const int prev = i == 0 ? -1 : keys[i - 1];
    const int cur = i == n ? nbuckets : keys[i];
    for (int c = prev + 1; c <= cur; c++) start[c] = (int32_t)i;
}

// Centres sorted by bucket (stable): perm, and the start of every bucket in it.  drop: centres outside an unclamped
// grid and dead beams are left out.  A window of steps binds this by its launches: the keys come with the counts of the first
// digit, the first pass makes its own indexes, and the buckets' bits are dealt evenly over the passes, which mostly
// keeps the counts short enough for the scan of one block: 7 launches where 13 were (8-bit digits, three scan kernels).  27 k
// beams, two windows: solve 0.745 -> 0.716 ms; layered population of 0.9 M, 60 samples: 18.9 -> 18.5 ms.
fga_status sort_centres(Workspace &ws, const BinGrid &g, const void *Q_src, int q_kind, int64_t q_stride, int64_t n,
                        const int32_t *cls_or_null, bool drop, int nbuckets, int32_t **perm_out, int32_t *cell_start,
                        int32_t *keys_copy, cudaStream_t s) {
    const size_t nn = (size_t)std::max<int64_t>(n, 1);
    FGA_TRY(ws.keys.ensure(sizeof(int32_t) * nn));
    FGA_TRY(ws.vals.ensure(sizeof(int32_t) * nn));
    *perm_out = ws.vals.as<int32_t>();
    uint32_t *count = nullptr;
    int32_t *ka = ws.keys.as<int32_t>(), *va = nullptr;
    if (n > 0) {
        FGA_TRY(ws.keys_alt.ensure(sizeof(int32_t) * nn));
        FGA_TRY(ws.vals_alt.ensure(sizeof(int32_t) * nn));
        int bits = 1;
        while ((1ll << bits) < (long long)nbuckets) bits++;
        const int passes = (bits + 7) / 8, db = (bits + passes - 1) / passes, digits = 1 << db;
        const int ntiles = (int)((n + RS_TILE - 1) / RS_TILE);
        const int64_t nh = (int64_t)digits * ntiles + 1;
        FGA_TRY(ws.hist.ensure(sizeof(uint32_t) * ((size_t)nh + 1)));
        uint32_t *hist = ws.hist.as<uint32_t>();
        count = hist + nh;
        int32_t *kb = ws.keys_alt.as<int32_t>(), *vb = ws.vals.as<int32_t>(), *vc = ws.vals_alt.as<int32_t>();
        for (int p = 0; p < passes; p++) {
            {
                ProfScope ps(P_BIN, s);
                if (p > 0)
                    rs_hist_kernel<<<ntiles, RS_T, 0, s>>>(ka, count, p * db, digits, ntiles, hist);
                else if (q_kind == Q_F32_AOS3)
                    keys_kernel<float><<<ntiles, RS_T, 0, s>>>(g, (const float *)Q_src, 3, 1, n, cls_or_null, drop, ka, digits,
                                                               ntiles, hist);
                else if (q_kind == Q_F32_SOA)
                    keys_kernel<float><<<ntiles, RS_T, 0, s>>>(g, (const float *)Q_src, 1, q_stride, n, cls_or_null, drop, ka,
                                                               digits, ntiles, hist);
                else
                    keys_kernel<double><<<ntiles, RS_T, 0, s>>>(g, (const double *)Q_src, 1, q_stride, n, cls_or_null, drop,
                                                                ka, digits, ntiles, hist);
            }
            FGA_CUDA(cudaGetLastError());
            if (p == 0 && keys_copy)
                FGA_CUDA(cudaMemcpyAsync(keys_copy, ka, sizeof(int32_t) * (size_t)n, cudaMemcpyDeviceToDevice, s));
            FGA_TRY(exclusive_scan(ws, hist, nh, s));
            ProfScope ps(P_BIN, s);
            rs_scatter_kernel<<<ntiles, RS_T, 0, s>>>(ka, va, n, count, p * db, digits, ntiles, hist, kb, vb);
            FGA_CUDA(cudaGetLastError());
            std::swap(ka, kb);
            va = vb;
            std::swap(vb, vc);
        }
        *perm_out = va;
    }
    ProfScope ps(P_BIN, s);
    cell_start_kernel<<<(unsigned)((n + 1 + 255) / 256), 256, 0, s>>>(ka, count, n, nbuckets, cell_start);
    FGA_CUDA(cudaGetLastError());
    return FGA_OK;
}

// ---------------------------------------------------------------------------------------------
// permutation of the beam state (sorted by cell, once per window of steps)
// ---------------------------------------------------------------------------------------------
template <typename R>
__global__ void permute_kernel(const R *__restrict__ src, R *__restrict__ dst, const int32_t *__restrict__ fsrc,
                               int32_t *__restrict__ fdst, const int32_t *__restrict__ isrc, int32_t *__restrict__ idst,
                               const int32_t *__restrict__ perm, int64_t n, int64_t cap) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const int64_t j = perm[i];
#pragma unroll 2
    for (int f = 0; f < NFS; f++) dst[(int64_t)f * cap + i] = src[(int64_t)f * cap + j];
    fdst[i] = fsrc[j];
    idst[i] = isrc[j];
}

fga_status permute_beams(fga_beams *b, const int32_t *perm, cudaStream_t s) {
    const size_t rb = b->precision == FGA_PREC_FP64 ? 8 : 4;
    FGA_TRY(b->state_alt.ensure(rb * NFS * b->cap));
    FGA_TRY(b->flags_alt.ensure(4 * b->cap));
    FGA_TRY(b->id_alt.ensure(4 * b->cap));
    const unsigned blocks = (unsigned)((b->nb + 255) / 256);
    if (b->nb > 0) {
        ProfScope ps(P_BIN, s);
        if (rb == 8)
            permute_kernel<double><<<blocks, 256, 0, s>>>(b->state.as<double>(), b->state_alt.as<double>(),
                                                          b->flags.as<int32_t>(), b->flags_alt.as<int32_t>(),
                                                          b->id.as<int32_t>(), b->id_alt.as<int32_t>(), perm, b->nb, b->cap);
        else
            permute_kernel<float><<<blocks, 256, 0, s>>>(b->state.as<float>(), b->state_alt.as<float>(),
                                                         b->flags.as<int32_t>(), b->flags_alt.as<int32_t>(),
                                                         b->id.as<int32_t>(), b->id_alt.as<int32_t>(), perm, b->nb, b->cap);
        FGA_CUDA(cudaGetLastError());
    }
    std::swap(b->state, b->state_alt);
    std::swap(b->flags, b->flags_alt);
    std::swap(b->id, b->id_alt);
    return FGA_OK;
}

// ---------------------------------------------------------------------------------------------
// Gaussian sum
// ---------------------------------------------------------------------------------------------
BinGrid make_grid(const double *pts, int64_t n, double reach) {
    double lo[3] = {1e300, 1e300, 1e300}, hi[3] = {-1e300, -1e300, -1e300};
    for (int64_t i = 0; i < n; i++)
        for (int d = 0; d < 3; d++) {
            lo[d] = std::min(lo[d], pts[3 * i + d]);
            hi[d] = std::max(hi[d], pts[3 * i + d]);
        }
    if (n == 0)
        for (int d = 0; d < 3; d++) lo[d] = hi[d] = 0.0;
    BinGrid g;
    const double h = reach * 1.001;  // slack for FP32 key rounding
    g.inv_h = (float)(1.0 / h);
    g.ncells = 1;
    for (int d = 0; d < 3; d++) {
        g.o[d] = (float)(lo[d] - reach * 1.0005);
        const double ext = hi[d] + reach * 1.0005 - (double)g.o[d];
        g.nc[d] = std::max(1, (int)std::ceil(ext * (double)g.inv_h));
        g.ncells *= g.nc[d];
    }
    g.clamp = false;
    return g;
}

// (beam, point) pairs that fell inside the window, counted when profiling is on
static __device__ unsigned long long g_pairs_in_window;

int64_t read_pair_counter(bool reset) {
    unsigned long long v = 0;
    if (cudaMemcpyFromSymbol(&v, g_pairs_in_window, sizeof v) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    if (reset) {
        const unsigned long long z = 0;
        cudaMemcpyToSymbol(g_pairs_in_window, &z, sizeof z);
    }
    return (int64_t)v;
}

// exp(am) (cos ph, sin ph) in FP64 by table (Tang's table-driven method: nearest table argument, a short Taylor series
// for the rest): SC_N angles and EX_N powers of two, residuals below pi/SC_N and ln 2/(2 EX_N), where the first omitted
// terms are 1e-18 of the result.  Table values carry the high word of their rounding error, so that sine, cosine and
// exponential are rounded once, as the library's: rms error 7.1e-17 of e^am for either (2 M arguments, |ph| to 1e6, am
// to -700).  28 FP64 operations; sincos and exp take 65.  Callers send |ph| > PH_MAX (the table index would leave its
// integer) and am < AM_MIN (near the smallest numbers) to the library functions.
constexpr int SC_N = 1024, EX_N = 1024;
constexpr double PH_MAX = 1e6, AM_MIN = -700.0;

struct GaussTables {
    double2 sc[SC_N];   // cos, sin of 2 pi i / SC_N
    double ex[EX_N];    // 2^(i / EX_N)
    int2 scl[SC_N];     // high words of what sc and ex round off
    int exl[EX_N];
};
static_assert(sizeof(GaussTables) % 16 == 0, "copied in 16-byte pieces");

static int rounding_word(long double x, double r) {
    const double d = (double)(x - (long double)r);
    int64_t u;
    std::memcpy(&u, &d, sizeof u);
    return (int)(u >> 32);
}

static const GaussTables &gauss_tables() {
    static const GaussTables *t = [] {
        auto *g = new GaussTables;
        const long double pi = 3.14159265358979323846264338327950288L;
        for (int i = 0; i < SC_N; i++) {
            // by octants, so that the zeros and the equal values come out exactly
            const int q = i / (SC_N / 4), j = i % (SC_N / 4);
            const bool up = j > SC_N / 8;
            const long double a = 2 * pi * (up ? SC_N / 4 - j : j) / SC_N;
            const long double c1 = up ? std::sin(a) : std::cos(a), s1 = up ? std::cos(a) : std::sin(a);
            const long double c = q == 0 ? c1 : q == 1 ? -s1 : q == 2 ? -c1 : s1, s = q == 0 ? s1 : q == 1 ? c1 : q == 2 ? -s1 : -c1;
            g->sc[i] = make_double2((double)c, (double)s);
            g->scl[i] = make_int2(rounding_word(c, (double)c), rounding_word(s, (double)s));
        }
        for (int i = 0; i < EX_N; i++) {
            const long double e = std::exp2((long double)i / EX_N);
            g->ex[i] = (double)e;
            g->exl[i] = rounding_word(e, (double)e);
        }
        return g;
    }();
    return *t;
}

__device__ __forceinline__ void gauss_phase_table(double ph, double am, const GaussTables &T, double *er, double *ei) {
    constexpr double ROUND = 6755399441055744.0;   // 1.5 * 2^52: the integer lands in the low word
    constexpr double TWO_PI = 6.283185307179586476925286766559, TWO_PI_LO = 2.4492935982947064e-16;
    constexpr double LN2 = 0.69314718055994530941723212145818, LN2_LO = 2.3190468138462996e-17;
    double t = fma(ph, SC_N / TWO_PI, ROUND);
    const int n = __double2loint(t) & (SC_N - 1);
    t -= ROUND;
    double r = fma(t, -TWO_PI / SC_N, ph);
    r = fma(t, -TWO_PI_LO / SC_N, r);
    const double r2 = r * r;
    const double cm = r2 * fma(r2, 1.0 / 24.0, -0.5);                       // cos r - 1
    const double sn = fma(r * r2, fma(r2, 1.0 / 120.0, -1.0 / 6.0), r);      // sin r
    const double2 A = T.sc[n];
    const int2 Al = T.scl[n];
    const double c = A.x + fma(-A.y, sn, fma(A.x, cm, __hiloint2double(Al.x, 0)));
    const double s = A.y + fma(A.x, sn, fma(A.y, cm, __hiloint2double(Al.y, 0)));
    t = fma(am, EX_N / LN2, ROUND);
    const int m = __double2loint(t);
    t -= ROUND;
    double q = fma(t, -LN2 / EX_N, am);
    q = fma(t, -LN2_LO / EX_N, q);
    const double p = fma(q * q, fma(q, fma(q, 1.0 / 24.0, 1.0 / 6.0), 0.5), q);   // exp q - 1
    double e = T.ex[m & (EX_N - 1)];
    e += fma(e, p, __hiloint2double(T.exl[m & (EX_N - 1)], 0));
    e = __hiloint2double(__double2hiint(e) + ((m >> 10) << 20), __double2loint(e));
    *er = e * c;
    *ei = e * s;
}
static_assert(EX_N == 1 << 10, "the power of two is the index above its table part");

// FP64: a warp takes 32 points of the tile and every fourth 32 of the item's beams, staged.  Bound by the FP64 pipe
// (a warp instruction in 16 cycles): 53 operations per pair, of which sine, cosine and exponential are 28 by table
// against about 65 of the library's.  With one beam at a time for all lanes 54% of the lanes were idle: outside its
// window, or without a point (scattered receivers are a few to a cell).  So a tile of n <= 16 points takes every point
// into 32/n' lanes (n' the power of two above), which share its beams and add their sums at the end in a fixed order,
// and an FP32 distance with a margin marks each lane's beams, of which it then takes its own next one.
// 0.37 M beams x 1,000 points, most of them within the window: 37.4 -> 27.1 ms (18.3 with compact tiles).
// The screen: beams and points relative to the tile's first point.  A pair inside the window has both within 3 rw of it
// (the points share a cell), so its FP32 distance is off by less than 2e-6 rw^2; the margin is 1e-5 rw^2.
constexpr int GD_WARPS = 4;
struct GatherF64Smem {
    GaussTables T;
    double rec[GD_WARPS][32][REC];   // then the warps' sums
    float q[GD_WARPS][32][3];
    unsigned npairs;
};

__global__ void __launch_bounds__(32 * GD_WARPS) gather_f64_kernel(const double *__restrict__ rec, int64_t rec_stride,
                                                                  const double *__restrict__ pts,
                                                                  const int32_t *__restrict__ tile_pts,
                                                                  const int4 *__restrict__ items, double k, double rw2,
                                                                  const GaussTables *__restrict__ tables,
                                                                  double *__restrict__ partial, int count_pairs) {
    extern __shared__ double2 gd_smem[];
    GatherF64Smem &S = *reinterpret_cast<GatherF64Smem *>(gd_smem);
    if (threadIdx.x == 0) S.npairs = 0;
    for (int i = threadIdx.x; i < (int)sizeof(GaussTables) / 16; i += 32 * GD_WARPS)
        reinterpret_cast<int4 *>(&S.T)[i] = reinterpret_cast<const int4 *>(tables)[i];
    __syncthreads();
    unsigned mine = 0;
    rec += blockIdx.y * rec_stride;
    const int4 it = items[blockIdx.x];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int pt = tile_pts[it.x * 32 + lane];   // the tile's points come first
    const int np = __popc(__ballot_sync(0xffffffffu, pt >= 0)), n2 = np <= 1 ? 1 : 1 << (32 - __clz(np - 1));
    const int pi = __shfl_sync(0xffffffffu, pt, lane & (n2 - 1)), p0 = __shfl_sync(0xffffffffu, pt, 0);
    // the lane's beams of a stage: j = lane / n2 mod 32 / n2
    const unsigned share = (n2 == 32   ? 0xffffffffu
                            : n2 == 16 ? 0x55555555u
                            : n2 == 8  ? 0x11111111u
                            : n2 == 4  ? 0x01010101u
                            : n2 == 2  ? 0x00010001u
                                       : 1u)
                           << (lane / n2);
    double x0, x1, x2;
    if (pi >= 0) {
        x0 = pts[3 * (int64_t)pi];
        x1 = pts[3 * (int64_t)pi + 1];
        x2 = pts[3 * (int64_t)pi + 2];
    } else {
        x0 = x1 = x2 = 1e30;
    }
    const double o0 = pts[3 * (int64_t)p0], o1 = pts[3 * (int64_t)p0 + 1], o2 = pts[3 * (int64_t)p0 + 2];
    const float f0 = (float)(x0 - o0), f1 = (float)(x1 - o1), f2 = (float)(x2 - o2);
    const float screen = fmaxf((float)(rw2 * 1.00001), 1e-37f);
    const int64_t b0 = it.y + 32 * warp, b1 = it.z;   // stages in turn: the warps' shares of the window are alike
    double acc[6] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
    const double hk = -0.5 * k;
    double(*R)[REC] = S.rec[warp];
    float(*Q)[3] = S.q[warp];
    for (int64_t b = b0; b < b1; b += 32 * GD_WARPS) {
        const int m = (int)min((int64_t)32, b1 - b);
        const double2 *src = reinterpret_cast<const double2 *>(rec + b * REC);
        __syncwarp();
#pragma unroll
        for (int j = 0; j < REC / 2; j++) {
            const int i = j * 32 + lane;
            if (i < m * (REC / 2)) reinterpret_cast<double2 *>(R)[i] = __ldg(src + i);
        }
        __syncwarp();
        if (lane < m) {
            Q[lane][0] = (float)(R[lane][0] - o0);
            Q[lane][1] = (float)(R[lane][1] - o1);
            Q[lane][2] = (float)(R[lane][2] - o2);
        }
        __syncwarp();
        unsigned mask = 0;
#pragma unroll 8
        for (int j = 0; j < m; j++) {
            const float g0 = f0 - Q[j][0], g1 = f1 - Q[j][1], g2 = f2 - Q[j][2];
            if (g0 * g0 + g1 * g1 + g2 * g2 <= screen) mask |= 1u << j;
        }
        mask &= share;
        while (mask) {
            const double *r = R[__ffs(mask) - 1];
            mask &= mask - 1;
            double q[REC];
#pragma unroll
            for (int j = 0; j < REC / 2; j++) {
                const double2 v = reinterpret_cast<const double2 *>(r)[j];
                q[2 * j] = v.x;
                q[2 * j + 1] = v.y;
            }
            const double d0 = x0 - q[0], d1 = x1 - q[1], d2 = x2 - q[2];
            const double r2 = d0 * d0 + d1 * d1 + d2 * d2;
            if (r2 <= rw2) {
                mine++;
                const double ph = k * (q[3] * d0 + q[4] * d1 + q[5] * d2), am = hk * r2;
                double er, ei;
                if (fabs(ph) <= PH_MAX && am >= AM_MIN)
                    gauss_phase_table(ph, am, S.T, &er, &ei);
                else
                    gauss_phase_exp<double>(ph, am, &er, &ei);
#pragma unroll
                for (int d = 0; d < 3; d++) cmac<double>(acc[2 * d], acc[2 * d + 1], q[6 + 2 * d], q[7 + 2 * d], er, ei);
            }
        }
    }
    __syncwarp();
    double *red = &S.rec[0][0][0];   // [warp][lane][12], a warp's own records
#pragma unroll
    for (int j = 0; j < 6; j++) {
        double v = acc[j];
        for (int o = n2; o < 32; o <<= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        red[(warp * 32 + lane) * REC + j] = pt >= 0 ? v : 0.0;
    }
    if (count_pairs) atomicAdd(&S.npairs, mine);
    __syncthreads();
    if (count_pairs && threadIdx.x == 0) atomicAdd(&g_pairs_in_window, (unsigned long long)S.npairs);
    if (warp == 0) {
#pragma unroll
        for (int j = 0; j < 6; j++) {
            double v[GD_WARPS];
#pragma unroll
            for (int w = 0; w < GD_WARPS; w++) v[w] = red[(w * 32 + lane) * REC + j];
            partial[(((int64_t)blockIdx.y * gridDim.x + blockIdx.x) * 32 + lane) * 6 + j] = (v[0] + v[1]) + (v[2] + v[3]);
        }
    }
}

// The same sum in FP32.  A warp takes 32 points of the tile and every fourth 32 of the item's beams.  Those whose window
// reaches the points' box are staged in shared memory field by field (the next 32 in flight in registers), so
// that two consecutive beams are the two halves of packed FP32x2 operands: coordinates and accumulators are packed
// once, and a pair of beams costs 30 packed FMAs, 6 MUFU and 12 other instructions for 64 (beam, point) pairs.  Bound
// by the FMA pipe (62 cycles a warp and 64 pairs; MUFU 48).  Against one beam and point per lane with uniform loads (41
// instructions per 32 pairs, long-scoreboard stalls): 1.05 M beams x 5,003 points 8.2 -> 5.3 ms, 100 samples of 256
// receivers and 1.05 M beams 43.0 -> 21.2 ms.  With compact tiles 4.20 and 21.2 ms, staging only what reaches the box
// 3.99 and 18.6 ms, the warps taking 32 beams in turn instead of a quarter of the item each 3.81 and 17.3 ms.
constexpr int GF_STAGE = 64;
struct alignas(16) GatherF32Stage {   // for its 16-byte reads (an array of floats alone is aligned to 4 bytes)
    float f[REC][GF_STAGE];
};
static_assert(alignof(GatherF32Stage) % sizeof(float4) == 0 && GF_STAGE * sizeof(float) % sizeof(float4) == 0 &&
              offsetof(GatherF32Stage, f) == 0, "16-byte reads of a field's beams");
__global__ void __launch_bounds__(128) gather_f32_kernel(const float *__restrict__ rec, int64_t rec_stride,
                                                         const double *__restrict__ pts,
                                                         const int32_t *__restrict__ tile_pts,
                                                         const int4 *__restrict__ items, float k, float rw2,
                                                         float *__restrict__ partial, int count_pairs) {
    __shared__ GatherF32Stage stage[4];
    __shared__ float red[4][32][6];
    __shared__ unsigned npairs;
    if (threadIdx.x == 0) npairs = 0;
    const int4 it = items[blockIdx.x];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int pi = tile_pts[it.x * 32 + lane];
    // padding lanes sit far away: no beam is in their window
    const float x0 = pi >= 0 ? (float)pts[3 * (int64_t)pi] : 1e15f, x1 = pi >= 0 ? (float)pts[3 * (int64_t)pi + 1] : 1e15f,
                x2 = pi >= 0 ? (float)pts[3 * (int64_t)pi + 2] : 1e15f;
    const float2 X0 = make_float2(x0, x0), X1 = make_float2(x1, x1), X2 = make_float2(x2, x2);
    const int64_t b0 = it.y + 32 * warp, b1 = it.z;   // 32 beams in turn: the warps' shares of the window are alike
    const float *r0 = rec + blockIdx.y * rec_stride;
    const float hk2 = -0.72134752044448170368f * k;   // -k/2 in units of log 2
    constexpr double TWO_PI = 6.283185307179586476925286766559;
    constexpr float TP_HI = (float)TWO_PI, TP_LO = (float)(TWO_PI - (double)TP_HI), INV_TP = (float)(1.0 / TWO_PI);
    constexpr float MAGIC = 12582912.f;   // 1.5 x 2^23: adding and subtracting it rounds to an integer
    auto bc = [](float v) { return make_float2(v, v); };
    float2 acc[6];
#pragma unroll
    for (int j = 0; j < 6; j++) acc[j] = bc(0.f);
    unsigned mine = 0;
    float4 n0, n1, n2;
    // lane's record of the 32 from b; a padding beam lies outside every window
    auto fetch = [&](int64_t b) {
        if (b + lane < b1) {
            const float4 *p = reinterpret_cast<const float4 *>(r0 + (b + lane) * REC);
            n0 = __ldg(p);
            n1 = __ldg(p + 1);
            n2 = __ldg(p + 2);
        } else {
            n0 = make_float4(-1e15f, -1e15f, -1e15f, 0.f);
            n1 = n2 = make_float4(0.f, 0.f, 0.f, 0.f);
        }
    };
    // the points' box: beams whose window does not reach it are not staged
    const float far = __int_as_float(0x7f800000);
    float lo[3] = {pi >= 0 ? x0 : far, pi >= 0 ? x1 : far, pi >= 0 ? x2 : far};
    float hi[3] = {pi >= 0 ? x0 : -far, pi >= 0 ? x1 : -far, pi >= 0 ? x2 : -far};
#pragma unroll
    for (int d = 0; d < 3; d++)
        for (int o = 16; o; o >>= 1) {
            lo[d] = fminf(lo[d], __shfl_xor_sync(0xffffffffu, lo[d], o));
            hi[d] = fmaxf(hi[d], __shfl_xor_sync(0xffffffffu, hi[d], o));
        }
    const float reach2 = fmaxf(rw2 * 1.00001f, 1e-37f);
    auto put = [&](int slot) {
        float *st = &stage[warp].f[0][slot];
        st[0 * GF_STAGE] = -n0.x;
        st[1 * GF_STAGE] = -n0.y;
        st[2 * GF_STAGE] = -n0.z;
        st[3 * GF_STAGE] = k * n0.w;
        st[4 * GF_STAGE] = k * n1.x;
        st[5 * GF_STAGE] = k * n1.y;
        st[6 * GF_STAGE] = n1.z;
        st[7 * GF_STAGE] = n1.w;
        st[8 * GF_STAGE] = n2.x;
        st[9 * GF_STAGE] = n2.y;
        st[10 * GF_STAGE] = n2.z;
        st[11 * GF_STAGE] = n2.w;
    };
    auto sum = [&](int first, int nb) {
        const float(*st)[GF_STAGE] = reinterpret_cast<const float(*)[GF_STAGE]>(&stage[warp].f[0][first]);
        for (int j = 0; j < nb; j += 4) {
            float4 f[6];
#pragma unroll
            for (int c = 0; c < 6; c++) f[c] = *reinterpret_cast<const float4 *>(&st[c][j]);
#pragma unroll
            for (int h = 0; h < 2; h++) {
                auto pr = [&](const float4 &v) { return h ? make_float2(v.z, v.w) : make_float2(v.x, v.y); };
                const float2 d0 = __fadd2_rn(X0, pr(f[0])), d1 = __fadd2_rn(X1, pr(f[1])), d2 = __fadd2_rn(X2, pr(f[2]));
                const float2 r2 = __ffma2_rn(d2, d2, __ffma2_rn(d1, d1, __fmul2_rn(d0, d0)));
                const bool in0 = r2.x <= rw2, in1 = r2.y <= rw2;
                if (!__any_sync(0xffffffffu, in0 || in1)) continue;
                mine += (in0 ? 1u : 0u) + (in1 ? 1u : 0u);
                const float2 ph = __ffma2_rn(pr(f[5]), d2, __ffma2_rn(pr(f[4]), d1, __fmul2_rn(pr(f[3]), d0)));
                // Cody-Waite reduction of the phase by 2 pi (two-part constant)
                const float2 n = __fadd2_rn(__ffma2_rn(ph, bc(INV_TP), bc(MAGIC)), bc(-MAGIC));
                const float2 r = __ffma2_rn(n, bc(-TP_LO), __ffma2_rn(n, bc(-TP_HI), ph));
                const float2 am = __fmul2_rn(r2, bc(hk2));
                float2 e, s, c;
                asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(e.x) : "f"(am.x));
                asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(e.y) : "f"(am.y));
                __sincosf(r.x, &s.x, &c.x);
                __sincosf(r.y, &s.y, &c.y);
                e.x = in0 ? e.x : 0.f;
                e.y = in1 ? e.y : 0.f;
                const float2 er = __fmul2_rn(e, c), ei = __fmul2_rn(e, s), mi = make_float2(-ei.x, -ei.y);
#pragma unroll
                for (int d = 0; d < 3; d++) {
                    const float2 ar = *reinterpret_cast<const float2 *>(&st[6 + 2 * d][j + 2 * h]);
                    const float2 ai = *reinterpret_cast<const float2 *>(&st[7 + 2 * d][j + 2 * h]);
                    acc[2 * d] = __ffma2_rn(ai, mi, __ffma2_rn(ar, er, acc[2 * d]));
                    acc[2 * d + 1] = __ffma2_rn(ai, er, __ffma2_rn(ar, ei, acc[2 * d + 1]));
                }
            }
        }
    };
    // the stage is a ring of two halves: a half is summed once it is full, the beams that follow fill the other
    int at = 0, pending = 0;
    fetch(b0);
    for (int64_t b = b0; b < b1; b += 128) {
        const float e0 = fmaxf(fmaxf(lo[0] - n0.x, n0.x - hi[0]), 0.f), e1 = fmaxf(fmaxf(lo[1] - n0.y, n0.y - hi[1]), 0.f),
                    e2 = fmaxf(fmaxf(lo[2] - n0.z, n0.z - hi[2]), 0.f);
        const bool keep = b + lane < b1 && e0 * e0 + e1 * e1 + e2 * e2 <= reach2;
        const unsigned kept = __ballot_sync(0xffffffffu, keep);
        if (keep) put((at + __popc(kept & ((1u << lane) - 1u))) & (GF_STAGE - 1));
        __syncwarp();
        if (b + 128 < b1) fetch(b + 128);
        const int nk = __popc(kept), half = (at - pending) & (GF_STAGE - 1);
        at = (at + nk) & (GF_STAGE - 1);
        pending += nk;
        if (pending >= GF_STAGE / 2) {
            sum(half, GF_STAGE / 2);
            pending -= GF_STAGE / 2;
        }
        __syncwarp();   // the half just read may be written next
    }
    if (pending > 0) {
        // up to three beams outside every window fill the last group of four
        if (lane < (-pending & 3)) {
            n0 = make_float4(-1e15f, -1e15f, -1e15f, 0.f);
            n1 = n2 = make_float4(0.f, 0.f, 0.f, 0.f);
            put((at + lane) & (GF_STAGE - 1));
        }
        __syncwarp();
        sum((at - pending) & (GF_STAGE - 1), pending);
    }
#pragma unroll
    for (int j = 0; j < 6; j++) red[warp][lane][j] = acc[j].x + acc[j].y;
    __syncthreads();
    if (count_pairs) {
        atomicAdd(&npairs, mine);
        __syncthreads();
        if (threadIdx.x == 0) atomicAdd(&g_pairs_in_window, (unsigned long long)npairs);
    }
    if (warp == 0) {
        float *dst = partial + (((int64_t)blockIdx.y * gridDim.x + blockIdx.x) * 32 + lane) * 6;
#pragma unroll
        for (int j = 0; j < 6; j++) dst[j] = (red[0][lane][j] + red[1][lane][j]) + (red[2][lane][j] + red[3][lane][j]);
    }
}

// The FP32 kernel multiplies the beams outside a lane's window by zero.  Where one of them has an infinite or NaN amplitude
// or phase the product is NaN, in points that the beam does not reach: an item's sums that are not finite are formed
// again by the reduction, one beam at a time and only into the lanes whose window holds it.  (Looking at every
// beam before it is staged cost 3.5% of the sum, a look at the sums at the end of the kernel 1.2 to 2.2%.)
__device__ __noinline__ void gather_f32_alone(const float *rec, int4 it, float x0, float x1, float x2, float k, float rw2,
                                              float *acc) {
    for (int j = 0; j < 6; j++) acc[j] = 0.f;
    for (int64_t b = it.y; b < it.z; b++) {
        const float *r = rec + b * REC;
        const float d0 = x0 - r[0], d1 = x1 - r[1], d2 = x2 - r[2], r2 = d0 * d0 + d1 * d1 + d2 * d2;
        if (r2 <= rw2) {
            float er, ei;
            gauss_phase_exp<float>(k * (r[3] * d0 + r[4] * d1 + r[5] * d2), -0.5f * k * r2, &er, &ei);
            for (int d = 0; d < 3; d++) cmac<float>(acc[2 * d], acc[2 * d + 1], r[6 + 2 * d], r[7 + 2 * d], er, ei);
        }
    }
}

// u at the points of a tile (blockIdx.x) and sample (blockIdx.y): RD_WARPS warps stride over the tile's items, then
// their FP64 sums are added in a fixed order.  (A single warp per tile walked thousands of items alone: 100 samples of
// 256 receivers and 1.05 M beams 17.0 -> 0.5 ms.)
constexpr int RD_WARPS = 16;
template <typename R>
__global__ void __launch_bounds__(32 * RD_WARPS) reduce_kernel(const R *__restrict__ partial,
                                                              const int32_t *__restrict__ tile_pts,
                                                              const int32_t *__restrict__ item_start, int nitems,
                                                              const R *__restrict__ rec, int64_t rec_stride,
                                                              const double *__restrict__ pts, const int4 *__restrict__ items,
                                                              R k, R rw2, R *__restrict__ u, int64_t u_stride) {
    __shared__ double sh[RD_WARPS][6][32];
    const int t = blockIdx.x, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int pi = tile_pts[t * 32 + lane];
    const R *p = partial + ((int64_t)blockIdx.y * nitems * 32 + lane) * 6;
    double acc[6] = {0, 0, 0, 0, 0, 0};
    for (int i = item_start[t] + warp; i < item_start[t + 1]; i += RD_WARPS) {
        R v[6];
#pragma unroll
        for (int j = 0; j < 6; j++) v[j] = p[(int64_t)i * 192 + j];
        if constexpr (sizeof(R) == 4) {
            const float zero = 0.f * ((v[0] + v[1]) + (v[2] + v[3]) + (v[4] + v[5]));
            if (pi >= 0 && !(zero == 0.f)) {
                float alone[6];
                gather_f32_alone(rec + blockIdx.y * rec_stride, items[i], (float)pts[3 * (int64_t)pi],
                                 (float)pts[3 * (int64_t)pi + 1], (float)pts[3 * (int64_t)pi + 2], k, rw2, alone);
#pragma unroll
                for (int j = 0; j < 6; j++) v[j] = alone[j];
            }
        }
#pragma unroll
        for (int j = 0; j < 6; j++) acc[j] += (double)v[j];
    }
#pragma unroll
    for (int j = 0; j < 6; j++) sh[warp][j][lane] = acc[j];
    __syncthreads();
    if (warp > 0 || pi < 0) return;
    R *dst = u + blockIdx.y * u_stride + (int64_t)pi * 6;
#pragma unroll
    for (int j = 0; j < 6; j++) {
#pragma unroll
        for (int w = 1; w < RD_WARPS; w++) acc[j] += sh[w][j][lane];
        dst[j] = (R)acc[j];
    }
}

fga_status build_sum_plan(Workspace &ws, const BinGrid &g, const int32_t *cell_start_dev, int nclasses,
                          const double *pts_host, int64_t npts, int samples, cudaStream_t s, SumPlan &plan) {
    plan.ntiles = 0;
    plan.nitems = 0;
    if (npts == 0) return FGA_OK;
    const int nbk = nclasses * (g.ncells + 1);
    FGA_TRY(ws.h_cell_start.ensure(sizeof(int32_t) * (size_t)(nbk + 1)));
    int32_t *cs = ws.h_cell_start.as<int32_t>();
    FGA_CUDA(cudaMemcpyAsync(cs, cell_start_dev, sizeof(int32_t) * (size_t)(nbk + 1), cudaMemcpyDeviceToHost, s));
    // points -> cells (host, FP64; the cell size carries slack for the FP32 beam keys)
    // A cell's points go into its tiles along a Morton curve over 8^3 parts of the cell: the points of a tile are close
    // together, so that a beam mostly lies in the window of all of them or of none and the kernels pass over it.  (In
    // the order given, a tile of scattered points spans its cell, and nearly every beam of the 27 cells, six times the
    // window's volume, met one of them: 1.05 M beams x 5,003 points 5.3 against 4.2 ms now, FP64, 0.37 M x 1,000 27.1
    // against 18.3 ms.)
    std::vector<int32_t> pcell((size_t)npts);
    std::vector<int64_t> key((size_t)npts);
    for (int64_t i = 0; i < npts; i++) {
        int c[3], m = 0;
        for (int d = 0; d < 3; d++) {
            const double t = (pts_host[3 * i + d] - (double)g.o[d]) * (double)g.inv_h;
            int cd = (int)std::floor(t);
            cd = std::min(std::max(cd, 0), g.nc[d] - 1);
            c[d] = cd;
            const int part = (int)std::min(7.0, std::max(0.0, 8.0 * (t - cd)));
            for (int bit = 0; bit < 3; bit++) m |= (part >> bit & 1) << (3 * bit + d);
        }
        pcell[(size_t)i] = (c[0] * g.nc[1] + c[1]) * g.nc[2] + c[2];
        key[(size_t)i] = (int64_t)pcell[(size_t)i] << 9 | m;
    }
    std::vector<int32_t> order((size_t)npts);
    std::iota(order.begin(), order.end(), 0);
    std::stable_sort(order.begin(), order.end(), [&](int32_t a, int32_t b) { return key[a] < key[b]; });
    std::vector<int32_t> tiles;  // 32 entries per tile
    std::vector<int32_t> tile_cell;
    for (int64_t i = 0; i < npts;) {
        const int cell = pcell[(size_t)order[(size_t)i]];
        int64_t j = i;
        while (j < npts && pcell[(size_t)order[(size_t)j]] == cell) j++;
        for (int64_t t0 = i; t0 < j; t0 += 32) {
            for (int l = 0; l < 32; l++) tiles.push_back(t0 + l < j ? order[(size_t)(t0 + l)] : -1);
            tile_cell.push_back(cell);
        }
        i = j;
    }
    const int ntiles = (int)tile_cell.size();
    FGA_CUDA(cudaStreamSynchronize(s));  // cell_start on the host
    plan.n_rec = 0;
    for (int cl = 0; cl < 4; cl++) {
        plan.n_in[cl] = 0;
        plan.rec_off[cl] = plan.n_rec;
        if (cl < nclasses) {
            const int cb = cl * (g.ncells + 1);
            plan.n_in[cl] = cs[cb + g.ncells] - cs[cb];
            plan.beg[cl] = cs[cb];
        }
        plan.n_rec += plan.n_in[cl];
    }
    // candidate ranges per tile: (c0 +- 1, c1 +- 1) x contiguous c2 - 1 .. c2 + 1, per class
    struct Rg {
        int tile, b, e;
    };
    std::vector<Rg> ranges;
    int64_t total = 0;
    for (int t = 0; t < ntiles; t++) {
        const int cell = tile_cell[(size_t)t];
        const int c2 = cell % g.nc[2], c1 = (cell / g.nc[2]) % g.nc[1], c0 = cell / (g.nc[2] * g.nc[1]);
        const int lo2 = std::max(c2 - 1, 0), hi2 = std::min(c2 + 1, g.nc[2] - 1);
        for (int cl = 0; cl < nclasses; cl++) {
            const int cb = cl * (g.ncells + 1);
            for (int a0 = std::max(c0 - 1, 0); a0 <= std::min(c0 + 1, g.nc[0] - 1); a0++)
                for (int a1 = std::max(c1 - 1, 0); a1 <= std::min(c1 + 1, g.nc[1] - 1); a1++) {
                    const int id0 = (a0 * g.nc[1] + a1) * g.nc[2];
                    // sorted positions -> compact record indices of class cl
                    const int64_t shift = plan.rec_off[cl] - cs[cb];
                    const int bb = (int)(cs[cb + id0 + lo2] + shift), ee = (int)(cs[cb + id0 + hi2 + 1] + shift);
                    if (ee > bb) {
                        ranges.push_back({t, bb, ee});
                        total += ee - bb;
                    }
                }
        }
    }
    // chunk size: work items of at least 512 beams, up to ~16384 of them for one sample (some 15 waves of the
    // ~1064 resident CTAs, so that the last wave's idle share is small: 4096 items are 6.2 waves, 5.73 against
    // 5.33 ms on 1.05 M beams x 5,003 points) and up to ~4096 a sample for several in one launch (fewer partial
    // sums: reductions of 100 samples 0.5 against 1.7 ms)
    const int64_t most = samples < 4 ? 16384 : 4096;
    int64_t B = std::max<int64_t>(512, (total + most - 1) / most);
    B = (B + 127) / 128 * 128;
    std::vector<int32_t> item_start((size_t)ntiles + 1, 0);
    std::vector<int4> items;
    size_t ri = 0;
    for (int t = 0; t < ntiles; t++) {
        item_start[(size_t)t] = (int32_t)items.size();
        while (ri < ranges.size() && ranges[ri].tile == t) {
            for (int64_t b = ranges[ri].b; b < ranges[ri].e; b += B)
                items.push_back(make_int4(t, (int)b, (int)std::min<int64_t>(b + B, ranges[ri].e), 0));
            ri++;
        }
    }
    item_start[(size_t)ntiles] = (int32_t)items.size();
    plan.ntiles = ntiles;
    plan.nitems = (int)items.size();
    const size_t tb = sizeof(int32_t) * tiles.size(), ib = sizeof(int4) * items.size(),
                 sb = sizeof(int32_t) * item_start.size();
    FGA_TRY(ws.tiles.ensure(tb + sb));
    FGA_TRY(ws.items.ensure(std::max<size_t>(ib, 16)));
    FGA_TRY(ws.h_tiles.ensure(tb + sb));
    FGA_TRY(ws.h_items.ensure(std::max<size_t>(ib, 16)));
    std::memcpy(ws.h_tiles.p, tiles.data(), tb);
    std::memcpy(static_cast<char *>(ws.h_tiles.p) + tb, item_start.data(), sb);
    if (ib) std::memcpy(ws.h_items.p, items.data(), ib);
    FGA_CUDA(cudaMemcpyAsync(ws.tiles.p, ws.h_tiles.p, tb + sb, cudaMemcpyHostToDevice, s));
    if (ib) FGA_CUDA(cudaMemcpyAsync(ws.items.p, ws.h_items.p, ib, cudaMemcpyHostToDevice, s));
    plan.tile_pts = ws.tiles.as<int32_t>();
    plan.item_start = reinterpret_cast<int32_t *>(static_cast<char *>(ws.tiles.p) + tb);
    plan.items = ws.items.as<int4>();
    plan.pairs_tested = total * 32;
    return FGA_OK;
}

fga_status run_sum(Workspace &ws, const SumPlan &plan, int precision, const void *rec, int64_t rec_stride, int ns,
                   const double *pts_dev, double k, double rw, void *u_out, int64_t u_stride, cudaStream_t s, int cat) {
    if (plan.ntiles == 0) return FGA_OK;
    const size_t rb = precision == FGA_PREC_FP64 ? 8 : 4;
    // as many samples per launch as keep the partial sums under SUM_PARTIAL_MAX bytes
    const size_t per_sample = rb * 32 * 6 * (size_t)std::max(plan.nitems, 1);
    int chunk = (int)std::max<size_t>(1, std::min<size_t>({(size_t)ns, SUM_PARTIAL_MAX / per_sample, 65535}));
    FGA_TRY(ensure_scratch(ws.partial, chunk, 1, [&](int c) { return per_sample * (size_t)c; }));
    GaussTables *tables = nullptr;
    if (rb == 8 && plan.nitems > 0) {
        FGA_TRY(ws.gauss_tables.ensure(sizeof(GaussTables)));
        tables = ws.gauss_tables.as<GaussTables>();
        FGA_CUDA(cudaMemcpyAsync(tables, &gauss_tables(), sizeof(GaussTables), cudaMemcpyHostToDevice, s));
    }
    const int cnt = prof_counting() ? 1 : 0;
    prof_add_pairs_tested(plan.pairs_tested * ns);
    for (int s0 = 0; s0 < ns; s0 += chunk) {
        const int m = std::min(chunk, ns - s0);
        if (plan.nitems > 0) {
            ProfScope ps(cat, s);
            const dim3 grid((unsigned)plan.nitems, (unsigned)m);
            if (rb == 8) {
                FGA_CUDA(cudaFuncSetAttribute(gather_f64_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                              (int)sizeof(GatherF64Smem)));
                gather_f64_kernel<<<grid, 32 * GD_WARPS, sizeof(GatherF64Smem), s>>>(
                    (const double *)rec + rec_stride * s0, rec_stride, pts_dev, plan.tile_pts, plan.items, k, rw * rw,
                    tables, ws.partial.as<double>(), cnt);
            } else {
                gather_f32_kernel<<<grid, 128, 0, s>>>((const float *)rec + rec_stride * s0, rec_stride, pts_dev,
                                                       plan.tile_pts, plan.items, (float)k, (float)(rw * rw),
                                                       ws.partial.as<float>(), cnt);
            }
            FGA_CUDA(cudaGetLastError());
        }
        ProfScope ps(P_REDUCE, s);
        const dim3 grid((unsigned)plan.ntiles, (unsigned)m);
        if (rb == 8)
            reduce_kernel<double><<<grid, 32 * RD_WARPS, 0, s>>>(ws.partial.as<double>(), plan.tile_pts, plan.item_start,
                                                                 plan.nitems, nullptr, 0, pts_dev, plan.items, k, rw * rw,
                                                                 (double *)u_out + u_stride * s0, u_stride);
        else
            reduce_kernel<float><<<grid, 32 * RD_WARPS, 0, s>>>(ws.partial.as<float>(), plan.tile_pts, plan.item_start,
                                                                plan.nitems, (const float *)rec + rec_stride * s0, rec_stride,
                                                                pts_dev, plan.items, (float)k, (float)(rw * rw),
                                                                (float *)u_out + u_stride * s0, u_stride);
        FGA_CUDA(cudaGetLastError());
    }
    return FGA_OK;
}

}  // namespace fga
