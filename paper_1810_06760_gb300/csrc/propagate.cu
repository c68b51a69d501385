// A3-A4: per-beam classical RK4 of the FGA ODEs, one thread per beam, the whole state in
// registers for all steps of a launch; reconstruction records written at sample times inside the
// launch's steps.
#include "fga_beam.cuh"
#include "cell_cache.cuh"
#include "straight.cuh"

#include <algorithm>

namespace fga {

// one record at index i of a buffer
template <typename R> __device__ __forceinline__ void store_record(R *__restrict__ rec, int64_t i, const R r[REC]) {
    // 48 or 96 bytes per record in 16-byte stores (the buffers are allocations of their own)
    if constexpr (sizeof(R) == 4) {
        float4 *dst = reinterpret_cast<float4 *>(rec + i * REC);
#pragma unroll
        for (int q = 0; q < 3; q++) dst[q] = make_float4(r[4 * q], r[4 * q + 1], r[4 * q + 2], r[4 * q + 3]);
    } else {
        double2 *dst = reinterpret_cast<double2 *>(rec + i * REC);
#pragma unroll
        for (int q = 0; q < 6; q++) dst[q] = make_double2(r[2 * q], r[2 * q + 1]);
    }
}
template <typename R> __device__ __forceinline__ float record_bound(const R r[REC]) {
    float m = 0.f;
#pragma unroll
    for (int q = 6; q < REC; q++) m = fmaxf(m, fabsf((float)r[q]));
    return m;
}
// a sample's bound of |A| entries: maximum over the converged lanes, one atomic by the lowest of them
// (non-negative floats order like their bit patterns; a NaN is left to the solve's check)
__device__ __forceinline__ void sample_bound(unsigned *amax, float m) {
    const unsigned mask = __activemask();
    const unsigned v = __reduce_max_sync(mask, m == m ? __float_as_uint(m) : 0u);
    if ((int)(threadIdx.x & 31) == __ffs(mask) - 1 && v) atomicMax(amax, v);
}

// out = x + h k over the NF state reals (FP32: pairs as packed FP32x2 FMAs)
template <typename R> __device__ __forceinline__ void axpy_state(R *out, const R *x, R h, const R *kv) {
    if constexpr (sizeof(R) == 4) {
        const float2 h2 = make_float2(h, h);
#pragma unroll
        for (int f = 0; f < NF; f += 2) {
            const float2 r = __ffma2_rn(h2, make_float2(kv[f], kv[f + 1]), make_float2(x[f], x[f + 1]));
            out[f] = r.x;
            out[f + 1] = r.y;
        }
    } else {
#pragma unroll
        for (int f = 0; f < NF; f++) out[f] = x[f] + h * kv[f];
    }
}

// the same without Q (fields 3 .. N-1)
template <int N> __device__ __forceinline__ void axpy_rest(float *out, const float *x, float h, const float *kv) {
    const float2 h2 = make_float2(h, h);
    out[3] = __fmaf_rn(h, kv[3], x[3]);
#pragma unroll
    for (int f = 4; f < N; f += 2) {
        const float2 r = __ffma2_rn(h2, make_float2(kv[f], kv[f + 1]), make_float2(x[f], x[f + 1]));
        out[f] = r.x;
        out[f + 1] = r.y;
    }
}

// One RHS evaluation per iteration of a single loop, so that the large right-hand side is compiled once
// (four inlined copies overflowed the instruction cache).  Classical RK4 with k1 = f(y_n):
//   e = 0: k2 = f(y + h/2 k1)   acc += h/3 k2,  tmp = y + h/2 k2
//   e = 1: k3 = f(tmp)          acc += h/3 k3,  tmp = y + h k3
//   e = 2: k4 = f(tmp)          acc += h/6 k4 (= y_{n+1}),  tmp = acc
//   e = 3: k1' = f(y_{n+1})     records of the step; y = acc, acc = y + h/6 k1', tmp = y + h/2 k1'
// Iteration -1 is an e = 3 without records: it forms k1 of the first step from y_0.
// The three Q entries of acc hold the step's increment instead (small numbers, rounded at their own
// scale); y_{n+1}'s Q is y_n's plus that increment by compensated summation (kahan_add).
template <typename R, int WAVE, int MED>
__global__ void __launch_bounds__(128) rk4_kernel(ModelDev M, R *__restrict__ st, const int32_t *__restrict__ flags,
                                                  int64_t cap, int64_t beg, int64_t n, R sg, R dt, int nsteps,
                                                  int n_samp, const int *__restrict__ samp_step,
                                                  const R *__restrict__ samp_theta, R w, R *__restrict__ rec,
                                                  int64_t rec_lim, int64_t rec_stride, unsigned *__restrict__ amax) {
    const int64_t b = beg + (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (b >= beg + n) return;
    R y[NF], acc[NF], tmp[NF], kk[NF], qc[3];
#pragma unroll
    for (int f = 0; f < NF; f++) {
        y[f] = st[(int64_t)f * cap + b];
        acc[f] = y[f];
        tmp[f] = y[f];
    }
#pragma unroll
    for (int d = 0; d < 3; d++) qc[d] = st[(int64_t)(F_QC + d) * cap + b];
    const bool ref_e1 = (flags[b] & FL_REF_E1) != 0;
    R s0[6];   // Q', P' at y_n (left slopes of the Hermite records)
    int js = 0;
    const R h2 = R(0.5) * dt, h3 = dt / R(3), h6 = dt / R(6);
    for (int it = -1; it < 4 * nsteps; it++) {
        const int e = it & 3;
        beam_rhs<R, WAVE, MED>(M, sg, ref_e1, tmp, kk);
        if (e == 3) {
            if (it >= 0) {
#pragma unroll
                for (int d = 0; d < 3; d++) {
                    R q = y[F_Q + d];
                    kahan_add<R>(q, qc[d], acc[F_Q + d]);
                    acc[F_Q + d] = q;       // acc = y_{n+1} in full
                }
            }
            const int step = it >> 2;
            while (it >= 0 && js < n_samp && samp_step[js] == step) {
                float mloc = 0.f;   // largest |A entry| of this thread's record
                if (b - beg < rec_lim) {
                    R r[REC];
                    beam_record6<R, WAVE>(ref_e1, y, s0, acc, kk, dt, samp_theta[js], w, r);
                    store_record<R>(rec, (int64_t)js * rec_stride + (b - beg), r);
                    mloc = record_bound<R>(r);
                }
                if (amax) sample_bound(amax + js, mloc);
                js++;
            }
#pragma unroll
            for (int f = 0; f < 6; f++) s0[f] = kk[f];
#pragma unroll
            for (int f = 0; f < NF; f++) y[f] = acc[f];
        }
        // acc += ca kk;  tmp = base + ct kk, base = y (e = 0, 1) or acc before its update (e = 2, 3; y for e = 3)
        const R ca = e < 2 ? h3 : h6;
        const R ct = e == 0 ? h2 : (e == 1 ? dt : (e == 2 ? h6 : h2));
        if (e < 2) {
            axpy_state<R>(tmp, y, ct, kk);
            axpy_state<R>(acc, acc, ca, kk);
        } else if (e == 2) {
            // tmp = y_{n+1} = y + (increment + h/6 k4) on Q
            axpy_state<R>(tmp, acc, ct, kk);
            axpy_state<R>(acc, acc, ca, kk);
#pragma unroll
            for (int d = 0; d < 3; d++) tmp[F_Q + d] = y[F_Q + d] + acc[F_Q + d];
        } else {
            axpy_state<R>(tmp, acc, ct, kk);
            axpy_state<R>(acc, acc, ca, kk);
#pragma unroll
            for (int d = 0; d < 3; d++) acc[F_Q + d] = ca * kk[F_Q + d];   // the new step's increment so far
        }
    }
#pragma unroll
    for (int f = 0; f < NF; f++) st[(int64_t)f * cap + b] = y[f];
#pragma unroll
    for (int d = 0; d < 3; d++) st[(int64_t)(F_QC + d) * cap + b] = qc[d];
}

// The classes' blocks of a beam set and of its records.
struct ClassBlocks {
    int64_t off[4], n[4];
    int64_t n_in[4], rec_off[4];
};

// Grid media, FP32: the same RK4 loop with the model sampled through the cell cache and the position of the
// next right-hand side formed as soon as this one's speed is known (the copies of new cells overlap with the rest
// of it).  One launch for all classes (blockIdx.y the class), so that small beam sets fill the SMs once instead of
// four times.  694 instructions per warp and right-hand side at 8 warps an SM (251 registers): the FMA pipe is
// 54% busy, the issue slots 59%, the L1 data pipe 53% on 0.44 M beams (rk4_kernel: 34%, 32%, 80% once the beams have spread).
// Propagation, 200 steps: 0.44 M beams 21.5 -> 10.8 ms, 2.7 M beams 108.4 -> 65.1 ms; 8.4 M beams x 100 steps with
// 250 samples 162 -> 112 ms.  Capped at 168 registers for 10 warps it spills: 113.6 ms on the 2.7 M beams.
template <int WAVE>
__device__ __forceinline__ void rk4_cell_body(const ModelDev &M, float *__restrict__ st, const int32_t *__restrict__ flags,
                                              int64_t cap, const ClassBlocks &cc, int cls, float dt, int nsteps,
                                              int n_samp, const int *__restrict__ samp_step,
                                              const float *__restrict__ samp_theta, float w, float *__restrict__ rec,
                                              int64_t rec_stride, unsigned *__restrict__ amax, float4 *smem) {
    const int64_t n = cc.n[cls];
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const int64_t b = cc.off[cls] + i;
    const float sg = (cls & 1) ? -1.f : 1.f;
    float y[NF], acc[NF], tmp[NF], kk[NF], qc[3];
#pragma unroll
    for (int f = 0; f < NF; f++) {
        y[f] = WAVE || f < F_A1 ? st[(int64_t)f * cap + b] : 0.f;   // a P beam has one amplitude
        acc[f] = y[f];
        tmp[f] = y[f];
    }
#pragma unroll
    for (int d = 0; d < 3; d++) qc[d] = st[(int64_t)(F_QC + d) * cap + b];
    const bool ref_e1 = (flags[b] & FL_REF_E1) != 0;
    CellCache cell;
    cell.init(WAVE ? M.gs : M.gp, smem);
    cell.prefetch(M, tmp);
    constexpr int NW = WAVE ? NF : F_A1;   // fields that change
    float s0[6];   // Q', P' at y_n (left slopes of the Hermite records)
    int js = 0;
    const float h2 = 0.5f * dt, h3 = dt / 3.f, h6 = dt / 6.f;
    for (int it = -1; it < 4 * nsteps; it++) {
        const int e = it & 3;
        float cf[10];
        cell.sample(cf);
        const float ca = e < 2 ? h3 : h6;
        const float ct = e == 0 ? h2 : (e == 1 ? dt : (e == 2 ? h6 : h2));
        // Q of the next right-hand side (tq) and of y_{n+1} (qn), as in rk4_kernel
        float tq[3], qn[3];
        {
            const float p2 = tmp[F_P] * tmp[F_P] + tmp[F_P + 1] * tmp[F_P + 1] + tmp[F_P + 2] * tmp[F_P + 2];
            const float ip = rsqrtf(p2), sc = sg * cf[0];
#pragma unroll
            for (int d = 0; d < 3; d++) {
                const float fq = sc * (tmp[F_P + d] * ip);
                if (e < 2) {
                    tq[d] = __fmaf_rn(ct, fq, y[F_Q + d]);
                    acc[F_Q + d] = __fmaf_rn(ca, fq, acc[F_Q + d]);
                } else if (e == 2) {
                    acc[F_Q + d] = __fmaf_rn(ca, fq, acc[F_Q + d]);
                    tq[d] = y[F_Q + d] + acc[F_Q + d];
                } else {
                    qn[d] = y[F_Q + d];
                    if (it >= 0) kahan_add<float>(qn[d], qc[d], acc[F_Q + d]);
                    tq[d] = __fmaf_rn(ct, fq, qn[d]);
                    acc[F_Q + d] = ca * fq;   // the new step's increment so far
                }
            }
        }
        if (it + 1 < 4 * nsteps) cell.prefetch(M, tq);
        beam_rhs_at<float, WAVE>(cf, sg, ref_e1, tmp, kk);
        if (e == 3) {
            const int step = it >> 2;
            while (it >= 0 && js < n_samp && samp_step[js] == step) {
                float mloc = 0.f;   // largest |A entry| of this thread's record
                if (i < cc.n_in[cls]) {
                    float y1[NF];   // y_{n+1}: acc with the compensated Q
#pragma unroll
                    for (int f = 0; f < NF; f++) y1[f] = f < 3 ? qn[f] : acc[f];
                    float r[REC];
                    beam_record6<float, WAVE>(ref_e1, y, s0, y1, kk, dt, samp_theta[js], w, r);
                    store_record<float>(rec, (int64_t)js * rec_stride + cc.rec_off[cls] + i, r);
                    mloc = record_bound<float>(r);
                }
                if (amax) sample_bound(amax + js, mloc);
                js++;
            }
#pragma unroll
            for (int f = 0; f < 6; f++) s0[f] = kk[f];
#pragma unroll
            for (int d = 0; d < 3; d++) y[F_Q + d] = qn[d];
#pragma unroll
            for (int f = 3; f < NF; f++) y[f] = acc[f];
        }
        // acc += ca kk;  tmp = base + ct kk, base = y (e = 0, 1) or acc before its update (e = 2, 3); Q is done
        if (e < 2)
            axpy_rest<NW>(tmp, y, ct, kk);
        else
            axpy_rest<NW>(tmp, acc, ct, kk);
        axpy_rest<NW>(acc, acc, ca, kk);
#pragma unroll
        for (int d = 0; d < 3; d++) tmp[F_Q + d] = tq[d];
    }
#pragma unroll
    for (int f = 0; f < NW; f++) st[(int64_t)f * cap + b] = y[f];
#pragma unroll
    for (int d = 0; d < 3; d++) st[(int64_t)(F_QC + d) * cap + b] = qc[d];
}

__global__ void __launch_bounds__(128) rk4_cell_kernel(ModelDev M, float *__restrict__ st, const int32_t *__restrict__ flags,
                                                      int64_t cap, ClassBlocks cc, float dt, int nsteps, int n_samp,
                                                      const int *__restrict__ samp_step,
                                                      const float *__restrict__ samp_theta, float w,
                                                      float *__restrict__ rec, int64_t rec_stride,
                                                      unsigned *__restrict__ amax) {
    extern __shared__ float4 cells[];
    const int cls = blockIdx.y;
    if (cls < 2)
        rk4_cell_body<0>(M, st, flags, cap, cc, cls, dt, nsteps, n_samp, samp_step, samp_theta, w, rec, rec_stride, amax,
                         cells);
    else
        rk4_cell_body<1>(M, st, flags, cap, cc, cls, dt, nsteps, n_samp, samp_step, samp_theta, w, rec, rec_stride, amax,
                         cells);
}

// Constant media: nsteps RK4 steps in closed form (straight.cuh), one launch for all classes
// (blockIdx.y the class).  Bound by the issue slots in FP32 (about 100 instructions a step, slots 86% used; the state's
// stream, 49 reals read and 28 written per beam and launch, is a quarter of the time) and by the FP64 pipe in FP64.  The
// steps gather the amplitudes' gain in one complex factor, applied at samples and at the end, and in FP64 two
// reciprocals share a division.  Against the general kernel's four right-hand sides per step: point-force experiment,
// 13.9 M beams x 79 steps FP32, 63.7 -> 3.8 ms; homogeneous experiment, 373 k beams x 100 steps FP64, 126.7 -> 7.7 ms
// (4.3 and 8.1 ms with both amplitudes advanced every step and a division per reciprocal).
template <typename R>
__global__ void __launch_bounds__(128) const_kernel(ModelDev M, R *__restrict__ st, const int32_t *__restrict__ flags,
                                                   int64_t cap, ClassBlocks cc, R dt, int nsteps, int n_samp,
                                                   const int *__restrict__ samp_step, const R *__restrict__ samp_theta,
                                                   R w, R *__restrict__ rec, int64_t rec_stride,
                                                   unsigned *__restrict__ amax) {
    const int cls = blockIdx.y, wave = cls >> 1;
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= cc.n[cls]) return;
    const int64_t b = cc.off[cls] + i;
    const R sg = (cls & 1) ? R(-1) : R(1);
    const R c = wave ? mp<R>(M.cs0, M.fcs0) : mp<R>(M.cp0, M.fcp0);
    R y[NF], qc[3], B[18];
#pragma unroll
    for (int f = 0; f < NF; f++) y[f] = st[(int64_t)f * cap + b];
#pragma unroll
    for (int d = 0; d < 3; d++) qc[d] = st[(int64_t)(F_QC + d) * cap + b];
    const bool ref_e1 = (flags[b] & FL_REF_E1) != 0;
    int js = 0;
    for (int n0 = 0; n0 < nsteps; n0 += STRAIGHT_RENEW) {
        Straight<R> S;
        straight_setup<R>(sg, c, y, B, S);
        const int m = min(STRAIGHT_RENEW, nsteps - n0);
        C2<R> g1 = straight_gamma<R>(S, R(0)), fac = {R(1), R(0)};   // fac: what the amplitudes have gained
        R rs = R(0);   // s, counted in FP64 (a conversion is an operation of the FP64 pipe)
        for (int s = 0; s < m; s++) {
            const R t = (sizeof(R) == 4 ? R(s) : rs) * dt;
            rs += R(1);
            C2<R> g2, g4;
            straight_gamma2<R>(S, t + R(0.5) * dt, t + dt, g2, g4);
            R y0[NF];   // Q, P and the amplitudes at the step's start (the rest is not read by a record)
#pragma unroll
            for (int f = 0; f < 6; f++) y0[f] = y[f];
            straight_q<R>(S, dt, y + F_Q, qc);
            const C2<R> f0 = fac, gain = straight_gain<R>(dt, g1, g2, g4), inc = cmul(gain, fac);
            fac = {fac.r + inc.r, fac.i + inc.i};
            g1 = g4;
            while (js < n_samp && samp_step[js] == n0 + s) {
                float mloc = 0.f;
                if (i < cc.n_in[cls]) {
                    const R sl[6] = {S.v[0], S.v[1], S.v[2], R(0), R(0), R(0)};
                    R r[REC], y1[NF];
#pragma unroll
                    for (int f = 0; f < 6; f++) y1[f] = y[f];
#pragma unroll
                    for (int f = F_A0; f < NF; f += 2) {
                        const C2<R> a = {y[f], y[f + 1]}, b0 = cmul(f0, a), b1 = cmul(fac, a);
                        y0[f] = b0.r;
                        y0[f + 1] = b0.i;
                        y1[f] = b1.r;
                        y1[f + 1] = b1.i;
                    }
                    if (wave)
                        beam_record6<R, 1>(ref_e1, y0, sl, y1, sl, dt, samp_theta[js], w, r);
                    else
                        beam_record6<R, 0>(ref_e1, y0, sl, y1, sl, dt, samp_theta[js], w, r);
                    store_record<R>(rec, (int64_t)js * rec_stride + cc.rec_off[cls] + i, r);
                    mloc = record_bound<R>(r);
                }
                if (amax) sample_bound(amax + js, mloc);
                js++;
            }
        }
#pragma unroll
        for (int f = F_A0; f < NF; f += 2) {
            const C2<R> a = cmul(fac, C2<R>{y[f], y[f + 1]});
            y[f] = a.r;
            y[f + 1] = a.i;
        }
        const R T = R(m) * dt;
#pragma unroll
        for (int f = 0; f < 18; f++) y[F_DQ + f] += T * B[f];
    }
#pragma unroll
    for (int f = 0; f < 3; f++) st[(int64_t)f * cap + b] = y[f];
#pragma unroll
    for (int f = F_DQ; f < F_DP; f++) st[(int64_t)f * cap + b] = y[f];
#pragma unroll
    for (int f = F_A0; f < NF; f++)
        if (f < F_A1 || wave) st[(int64_t)f * cap + b] = y[f];   // a P beam has one amplitude
#pragma unroll
    for (int d = 0; d < 3; d++) st[(int64_t)(F_QC + d) * cap + b] = qc[d];
}

// records of the current state (theta = 0), gathered in the order of perm (or identity)
template <typename R, int WAVE>
__global__ void records_kernel(const R *__restrict__ st, const int32_t *__restrict__ flags, int64_t cap,
                               const int32_t *__restrict__ perm, int64_t beg, int64_t n, R w, R *__restrict__ rec) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const int64_t b = perm ? perm[beg + i] : beg + i;
    R y[NF];
#pragma unroll
    for (int f = 0; f < NF; f++) y[f] = st[(int64_t)f * cap + b];
#pragma unroll
    for (int d = 0; d < 3; d++) y[F_Q + d] -= st[(int64_t)(F_QC + d) * cap + b];   // compensated Q
    R r[REC];
    beam_record<R, WAVE>((flags[b] & FL_REF_E1) != 0, y, y, y, y, R(0), R(0), w, r);
    store_record<R>(rec, i, r);
}

template <typename R, int WAVE, int MED>
static void launch_one(const fga_model *m, fga_beams *b, int cls, R dt, int nsteps, const SampleWindow *sw,
                       cudaStream_t s) {
    const int64_t n = b->n_cls[cls];
    if (n == 0) return;
    const int T = 128;
    const int64_t blocks = (n + T - 1) / T;
    const R sg = (cls & 1) ? R(-1) : R(1);
    R *rec = sw ? static_cast<R *>(sw->rec) + sw->rec_off[cls] * REC : nullptr;
    prof_add_beam_steps(n * (int64_t)nsteps);
    ProfScope ps(P_PROP, s);
    rk4_kernel<R, WAVE, MED><<<(unsigned)blocks, T, 0, s>>>(
        m->dev, b->state.as<R>(), b->flags.as<int32_t>(), b->cap, b->off_cls[cls], n, sg, dt, nsteps,
        sw ? sw->n : 0, sw ? sw->step : nullptr, sw ? static_cast<const R *>(sw->theta) : nullptr, (R)b->w, rec,
        sw ? sw->n_in[cls] : 0, sw ? sw->n_rec : 0, (sw && sizeof(R) == 4) ? sw->amax : nullptr);
}

template <typename R, int MED>
static void launch_med(const fga_model *m, fga_beams *b, R dt, int nsteps, const SampleWindow *sw, cudaStream_t s) {
    for (int cls = 0; cls < 4; cls++) {
        if (cls < 2)
            launch_one<R, 0, MED>(m, b, cls, dt, nsteps, sw, s);
        else
            launch_one<R, 1, MED>(m, b, cls, dt, nsteps, sw, s);
    }
}

static ClassBlocks class_blocks(const fga_beams *b, const SampleWindow *sw, int64_t *most) {
    ClassBlocks cc{};
    *most = 0;
    for (int c = 0; c < 4; c++) {
        cc.off[c] = b->off_cls[c];
        cc.n[c] = b->n_cls[c];
        cc.n_in[c] = sw ? sw->n_in[c] : 0;
        cc.rec_off[c] = sw ? sw->rec_off[c] : 0;
        *most = std::max(*most, cc.n[c]);
    }
    return cc;
}

template <typename R>
static void launch_const(const fga_model *m, fga_beams *b, R dt, int nsteps, const SampleWindow *sw, cudaStream_t s) {
    int64_t most;
    const ClassBlocks cc = class_blocks(b, sw, &most);
    if (most == 0) return;
    prof_add_beam_steps(b->nb * (int64_t)nsteps);
    ProfScope ps(P_PROP, s);
    const dim3 grid((unsigned)((most + 127) / 128), 4);
    const_kernel<R><<<grid, 128, 0, s>>>(m->dev, b->state.as<R>(), b->flags.as<int32_t>(), b->cap, cc, dt, nsteps,
                                         sw ? sw->n : 0, sw ? sw->step : nullptr,
                                         sw ? static_cast<const R *>(sw->theta) : nullptr, (R)b->w,
                                         sw ? static_cast<R *>(sw->rec) : nullptr, sw ? sw->n_rec : 0,
                                         (sw && sizeof(R) == 4) ? sw->amax : nullptr);
}

static fga_status launch_grid_f32(const fga_model *m, fga_beams *b, float dt, int nsteps, const SampleWindow *sw,
                                  cudaStream_t s) {
    int64_t most;
    const ClassBlocks cc = class_blocks(b, sw, &most);
    if (most == 0) return FGA_OK;
    prof_add_beam_steps(b->nb * (int64_t)nsteps);
    ProfScope ps(P_PROP, s);
    const dim3 grid((unsigned)((most + 127) / 128), 4);
    const int smem = 128 * CELL_STRIDE * (int)sizeof(float4);
    FGA_CUDA(cudaFuncSetAttribute(rk4_cell_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
    rk4_cell_kernel<<<grid, 128, smem, s>>>(m->dev, b->state.as<float>(), b->flags.as<int32_t>(), b->cap, cc, dt, nsteps,
                                            sw ? sw->n : 0, sw ? sw->step : nullptr,
                                            sw ? static_cast<const float *>(sw->theta) : nullptr, (float)b->w,
                                            sw ? static_cast<float *>(sw->rec) : nullptr, sw ? sw->n_rec : 0,
                                            sw ? sw->amax : nullptr);
    return FGA_OK;
}

template <typename R>
static void launch_prec(const fga_model *m, fga_beams *b, R dt, int nsteps, const SampleWindow *sw, cudaStream_t s) {
    switch (m->dev.kind) {
    case FGA_MEDIUM_CONST: launch_const<R>(m, b, dt, nsteps, sw, s); break;
    case FGA_MEDIUM_SINE: launch_med<R, FGA_MEDIUM_SINE>(m, b, dt, nsteps, sw, s); break;
    case FGA_MEDIUM_GRID:
        // FP32 grid media take launch_grid_f32
        if constexpr (sizeof(R) == 8) launch_med<R, FGA_MEDIUM_GRID>(m, b, dt, nsteps, sw, s);
        break;
    default: break;   // layered media advance by launch_layered_steps
    }
}

fga_status launch_propagate(const fga_model *m, fga_beams *b, double dt, int nsteps, const SampleWindow *sw,
                            cudaStream_t s) {
    if (nsteps <= 0 && (!sw || sw->n == 0)) return FGA_OK;
    if (b->precision == FGA_PREC_FP64)
        launch_prec<double>(m, b, dt, nsteps, sw, s);
    else if (m->dev.kind == FGA_MEDIUM_GRID)
        FGA_TRY(launch_grid_f32(m, b, (float)dt, nsteps, sw, s));
    else
        launch_prec<float>(m, b, (float)dt, nsteps, sw, s);
    FGA_CUDA(cudaGetLastError());
    return FGA_OK;
}

fga_status launch_records_from_state(const fga_beams *b, const int32_t *perm, const int64_t beg[4],
                                     const int64_t n_in[4], const int64_t rec_off[4], void *rec, cudaStream_t s) {
    const int T = 256;
    for (int cls = 0; cls < 4; cls++) {
        const int64_t nc = n_in[cls];
        if (nc == 0) continue;
        const unsigned blocks = (unsigned)((nc + T - 1) / T);
        ProfScope ps(P_REC, s);
        if (b->precision == FGA_PREC_FP64) {
            double *dst = (double *)rec + rec_off[cls] * REC;
            if (cls < 2)
                records_kernel<double, 0><<<blocks, T, 0, s>>>(b->state.as<double>(), b->flags.as<int32_t>(), b->cap,
                                                               perm, beg[cls], nc, b->w, dst);
            else
                records_kernel<double, 1><<<blocks, T, 0, s>>>(b->state.as<double>(), b->flags.as<int32_t>(), b->cap,
                                                               perm, beg[cls], nc, b->w, dst);
        } else {
            float *dst = (float *)rec + rec_off[cls] * REC;
            if (cls < 2)
                records_kernel<float, 0><<<blocks, T, 0, s>>>(b->state.as<float>(), b->flags.as<int32_t>(), b->cap,
                                                              perm, beg[cls], nc, (float)b->w, dst);
            else
                records_kernel<float, 1><<<blocks, T, 0, s>>>(b->state.as<float>(), b->flags.as<int32_t>(), b->cap,
                                                              perm, beg[cls], nc, (float)b->w, dst);
        }
    }
    FGA_CUDA(cudaGetLastError());
    return FGA_OK;
}

}  // namespace fga
