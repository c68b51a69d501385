// A1-A2: wave-packet (FBI) transform of the initial data (Eq. psi) as three per-axis complex
// contractions, then beam initialisation (Eqs. alpha^k, ini_plus/ini_minus, op_zZ_app).
#include <algorithm>
#include <cmath>
#include <cstring>
#include <type_traits>

#include "fga_beam.cuh"
#include "gather.cuh"
#include "tc_gemm.cuh"

namespace fga {

// per-axis kernel K[a][i] = exp(-i k p (y_i - q) - k (y_i - q)^2 / 2), a = iq * np + jp
template <typename R>
__global__ void fbi_axis_kernel(C2<R> *__restrict__ K, int nq, int np, int ny, double q0, double dq, double p0,
                                double dp, double y0, double dy, double k) {
    const int idx = blockIdx.x * blockDim.x + threadIdx.x;
    const int A = nq * np;
    if (idx >= A * ny) return;
    const int a = idx / ny, i = idx % ny;
    const int iq = a / np, jp = a % np;
    const double q = q0 + iq * dq, p = p0 + jp * dp, y = y0 + i * dy;
    const double d = y - q;
    double s, c;
    sincos(-k * p * d, &s, &c);
    const double e = exp(-0.5 * k * d * d);
    K[idx] = {(R)(e * c), (R)(e * s)};
}

template <typename R> __device__ __forceinline__ C2<R> to_c2(const double2 v) { return {(R)v.x, (R)v.y}; }
template <typename R> __device__ __forceinline__ C2<R> to_c2(const C2<R> v) { return v; }

// Batched strided complex GEMM: C[z][m][n] = scale * sum_k A[z][m][k] B[n][k].
// A elements of type TA (complex128 input or R intermediates), B and C of type R.
// FP64, bound by the FP64 pipe (a warp instruction in 16 cycles, so shared-memory loads and occupancy are no concern):
// what counts is that no tile holds padding and that the SMs get equal shares.  A thread takes one row and J columns,
// a block 32 x 8 J; the launch takes the J that pads N least.  A complex product is four FMAs in chains (acc + (a b - c d)
// as written is a product, an FMA and an addition: six).  N = 72, K = 96, the three stages: 64 x 64 tiles (two, 44%
// padding) with six operations 20.6 ms, this 6.5 ms.
template <typename R, typename TA, int J>
__global__ void __launch_bounds__(256) cgemm_kernel(const TA *__restrict__ A, int64_t sAz, int64_t sAm, int64_t sAk,
                                                    const C2<R> *__restrict__ B, int64_t sBn, int64_t sBk,
                                                    C2<R> *__restrict__ Cm, int64_t sCz, int64_t sCm, int64_t sCn,
                                                    int64_t M, int N, int K, R scale) {
    constexpr int TM = 32, TN = 8 * J, TK = 16;
    __shared__ C2<R> As[TK][TM + 1];
    __shared__ C2<R> Bs[TK][TN + 1];
    const int z = blockIdx.z;
    const int64_t m0 = (int64_t)blockIdx.x * TM;
    const int n0 = blockIdx.y * TN;
    const int tx = threadIdx.x % 32, ty = threadIdx.x / 32;
    C2<R> acc[J];
#pragma unroll
    for (int j = 0; j < J; j++) acc[j] = {R(0), R(0)};
    const TA *Az = A + z * sAz;
    for (int k0 = 0; k0 < K; k0 += TK) {
        for (int e = threadIdx.x; e < TK * TM; e += 256) {
            const int mm = e % TM, kk = e / TM;
            const int64_t gm = m0 + mm;
            const int gk = k0 + kk;
            C2<R> v = {R(0), R(0)};
            if (gm < M && gk < K) v = to_c2<R>(Az[gm * sAm + (int64_t)gk * sAk]);
            As[kk][mm] = v;
        }
        for (int e = threadIdx.x; e < TK * TN; e += 256) {
            const int kk = e % TK, nn = e / TK;
            const int gn = n0 + nn, gk = k0 + kk;
            Bs[kk][nn] = (gn < N && gk < K) ? B[(int64_t)gn * sBn + (int64_t)gk * sBk] : C2<R>{R(0), R(0)};
        }
        __syncthreads();
#pragma unroll
        for (int kk = 0; kk < TK; kk++) {
            const C2<R> a = As[kk][tx];
#pragma unroll
            for (int j = 0; j < J; j++) {
                const C2<R> b = Bs[kk][ty + 8 * j];
                cmac<R>(acc[j].r, acc[j].i, a.r, a.i, b.r, b.i);
            }
        }
        __syncthreads();
    }
    const int64_t gm = m0 + tx;
    if (gm >= M) return;
#pragma unroll
    for (int j = 0; j < J; j++) {
        const int gn = n0 + ty + 8 * j;
        if (gn < N) Cm[z * sCz + gm * sCm + (int64_t)gn * sCn] = {acc[j].r * scale, acc[j].i * scale};
    }
}

template <typename R, typename TA>
static fga_status cgemm(const TA *A, int64_t sAz, int64_t sAm, int64_t sAk, const C2<R> *B, int64_t sBn, int64_t sBk,
                        C2<R> *Cm, int64_t sCz, int64_t sCm, int64_t sCn, int Z, int64_t M, int N, int K, R scale,
                        cudaStream_t s) {
    int J = 9, least = 1 << 30;
    for (int j = 9; j >= 2; j--) {
        const int padded = (N + 8 * j - 1) / (8 * j) * 8 * j;
        if (padded < least) {
            least = padded;
            J = j;
        }
    }
    dim3 grid((unsigned)((M + 31) / 32), (unsigned)((N + 8 * J - 1) / (8 * J)), (unsigned)Z);
    ProfScope ps(P_DECOMP, s);
    auto go = [&](auto jc) {
        cgemm_kernel<R, TA, decltype(jc)::value>
            <<<grid, 256, 0, s>>>(A, sAz, sAm, sAk, B, sBn, sBk, Cm, sCz, sCm, sCn, M, N, K, scale);
    };
    using std::integral_constant;
    switch (J) {
    case 2: go(integral_constant<int, 2>{}); break;
    case 3: go(integral_constant<int, 3>{}); break;
    case 4: go(integral_constant<int, 4>{}); break;
    case 5: go(integral_constant<int, 5>{}); break;
    case 6: go(integral_constant<int, 6>{}); break;
    case 7: go(integral_constant<int, 7>{}); break;
    case 8: go(integral_constant<int, 8>{}); break;
    default: go(integral_constant<int, 9>{}); break;
    }
    FGA_CUDA(cudaGetLastError());
    return FGA_OK;
}

// F[a0][a1][a2][c] = dy^3 sum_y f[y0][y1][y2][c] K0[a0][y0] K1[a1][y1] K2[a2][y2]
// The three stages (contract y2, then y1, then y0) are batched strided complex GEMMs: on the tensor
// cores (FP16 split, FP32 accumulation) for the FP32 path, on the FP64 pipe for the FP64 path.
struct TransformScratch {
    float *amax = nullptr;   // DEVICE: max |Re|, |Im| of the input
    int *err = nullptr;      // DEVICE: set by a tensor-core wait that ran out
    double S[3] = {1, 1, 1}; // max over kernel rows of sum_i |K_d[a][i]| per axis (bounds of the stages)
};

static fga_status fbi_transform_f64(const fga_init_desc *d, const double2 *f, C2<double> *const Kax[3], C2<double> *T1,
                                    C2<double> *T2, C2<double> *F, cudaStream_t s) {
    using D2 = C2<double>;
    const int A = d->nq * d->np;
    const int n0 = d->ny[0], n1 = d->ny[1], n2 = d->ny[2];
    // stage 1 (contract y2), one GEMM per component c: T1[(y0,y1)][a2][c]
    FGA_TRY((cgemm<double, double2>(f, 1, (int64_t)n2 * 3, 3, Kax[2], n2, 1, T1, 1, (int64_t)A * 3, 3, 3, (int64_t)n0 * n1,
                                    A, n2, 1.0, s)));
    // stage 2 (contract y1): T2[y0][a1][(a2,c)] ; batch y0, m = (a2,c), n = a1, k = y1
    FGA_TRY((cgemm<double, D2>(T1, (int64_t)n1 * A * 3, 1, (int64_t)A * 3, Kax[1], n1, 1, T2, (int64_t)A * A * 3, 1,
                               (int64_t)A * 3, n0, (int64_t)A * 3, A, n1, 1.0, s)));
    // stage 3 (contract y0): F[a0][(a1,a2,c)], m = (a1,a2,c), n = a0, k = y0
    const double vol = d->dy[0] * d->dy[1] * d->dy[2];
    return cgemm<double, D2>(T2, 0, 1, (int64_t)A * A * 3, Kax[0], n0, 1, F, 0, 1, (int64_t)A * A * 3, 1,
                             (int64_t)A * A * 3, A, n0, vol, s);
}

// the same on the tensor cores; stage 1 takes the components as rows (m = 3 (y0,y1) + c), so that the data are read
// in one pass
static fga_status fbi_transform_f32(const fga_init_desc *d, const double2 *f, const KernelMatrices &K, float2 *T1,
                                    float2 *T2, float2 *F, const TransformScratch &ts, cudaStream_t s) {
    const int A = d->nq * d->np;
    const int n0 = d->ny[0], n1 = d->ny[1], n2 = d->ny[2];
    const int64_t A3 = (int64_t)A * 3;
    FGA_TRY(tc_absmax(f, (int64_t)n0 * n1 * n2 * 3, ts.amax, s));
    // |Re|, |Im| of a stage's output <= sqrt(2) max(|Re|, |Im|) of its input x sum_i |K[a][i]|
    const double g1 = std::sqrt(2.0) * ts.S[2], g2 = g1 * std::sqrt(2.0) * ts.S[1];
    FGA_TRY((tc_cgemm<double2>(f, 0, (int64_t)n2 * 3, 3, K.ax[2], T1, 0, A3, 3, 3, 1, (int64_t)n0 * n1 * 3, A, 1.f, ts.amax,
                               1.f, ts.err, s)));
    FGA_TRY((tc_cgemm<float2>(T1, n1 * A3, 1, A3, K.ax[1], T2, A * A3, 1, A3, 1, n0, A3, A, 1.f, ts.amax, (float)g1, ts.err,
                              s)));
    const float vol = (float)(d->dy[0] * d->dy[1] * d->dy[2]);
    return tc_cgemm<float2>(T2, 0, 1, A * A3, K.ax[0], F, 0, 1, A * A3, 1, 1, A * A3, A, vol, ts.amax, (float)g2, ts.err, s);
}

// max over the q nodes of sum_i exp(-k (y_i - q)^2 / 2): the largest row sum of |K| on one axis
static double kernel_row_sum_max(int nq, double q0, double dq, int ny, double y0, double dy, double k) {
    double best = 0.0;
    for (int iq = 0; iq < nq; iq++) {
        const double q = q0 + iq * dq;
        double sum = 0.0;
        for (int i = 0; i < ny; i++) {
            const double t = y0 + i * dy - q;
            sum += std::exp(-0.5 * k * t * t);
        }
        best = std::max(best, sum);
    }
    return best;
}

struct MeshIndex {
    int q[3], p[3];
    int64_t f;   // of F's first component at the point
};

__device__ __forceinline__ MeshIndex mesh_index(int nq, int np, uint32_t mi) {
    const uint32_t p1 = (uint32_t)np, q1 = (uint32_t)nq;
    MeshIndex x;
    uint32_t t = mi / p1;
    x.p[2] = (int)(mi - t * p1);
    uint32_t u = t / p1;
    x.p[1] = (int)(t - u * p1);
    t = u / p1;
    x.p[0] = (int)(u - t * p1);
    u = t / q1;
    x.q[2] = (int)(t - u * q1);
    t = u / q1;
    x.q[1] = (int)(u - t * q1);
    x.q[0] = (int)t;
    const int A = nq * np;
    x.f = (((int64_t)(x.q[0] * np + x.p[0]) * A + (x.q[1] * np + x.p[1])) * A + (x.q[2] * np + x.p[2])) * 3;
    return x;
}

__device__ __forceinline__ double axis_node(double3 o, double3 d, int axis, int i) {
    const double a = axis == 0 ? o.x : axis == 1 ? o.y : o.z, h = axis == 0 ? d.x : axis == 1 ? d.y : d.z;
    return a + i * h;
}

// initial amplitudes (2^{3/2} psi, two components) and flags of the beam at q, p (qd: q in FP64, read in layered media
// only) of class cls
template <typename R, int MED>
__device__ __forceinline__ void beam_amplitudes(const ModelDev &Md, const C2<R> *__restrict__ F,
                                                const C2<R> *__restrict__ G, int64_t fidx, const double *qd, const R *q,
                                                const R *p, double k, int cls, R *amp, int &fl) {
    const int wave = cls >= 2;
    R cf[10];
    // layered media: the layer of q from its depth along the layer normal (x3 unless the layers are tilted),
    // minus its distance to the centre of spherical layers, or the undulating interfaces at or above it;
    // c(q) is that layer's speed
    int lay = 0;
    if (MED == FGA_MEDIUM_LAYERED) {
        if (Md.undul) {
            const double cc = cos(Md.uk[0] * qd[0]) * cos(Md.uk[1] * qd[1]);
            for (int l = 0; l < Md.nlay - 1; l++) lay += (qd[2] >= Md.zif[l] + Md.uamp[l] * cc) ? 1 : 0;
        } else {
            double zl = qd[2];
            if (Md.shells) {
                const double r0 = qd[0] - Md.ctr[0], r1 = qd[1] - Md.ctr[1], r2 = qd[2] - Md.ctr[2];
                zl = -sqrt(r0 * r0 + r1 * r1 + r2 * r2);
            } else if (Md.tilted) {
                zl = Md.R[6] * qd[0] + Md.R[7] * qd[1] + Md.R[8] * qd[2];
            }
            for (int l = 0; l < Md.nlay - 1; l++) lay += (zl >= Md.zif[l]) ? 1 : 0;
        }
        cf[0] = wave ? mp<R>(Md.lcs[lay], Md.flcs[lay]) : mp<R>(Md.lcp[lay], Md.flcp[lay]);
        for (int f = 1; f < 10; f++) cf[f] = R(0);
    } else {
        model_eval<R, MED>(Md, wave, q, cf);
    }
    const R pn = Real<R>::sqrt_(p[0] * p[0] + p[1] * p[1] + p[2] * p[2]);
    const R sgn = (cls & 1) ? R(-1) : R(1);
    const R gsc = sgn / ((R)k * cf[0] * pn);  // +- 1/(k c(q) |p|)
    R dirs[2][3];
    int nd = 1;
    fl = cls;
    if (!wave) {
        for (int d = 0; d < 3; d++) dirs[0][d] = p[d] / pn;
    } else {
        const bool r1 = (p[0] * p[0] + p[1] * p[1]) < R(0.01) * pn * pn;
        if (r1) fl |= FL_REF_E1;
        s_frame<R>(p, r1, dirs[0], dirs[1]);
        nd = 2;
    }
    const R a0 = R(2.8284271247461900976033774484194);  // 2^{3/2}
    for (int j = 0; j < 4; j++) amp[j] = R(0);
    for (int j = 0; j < nd; j++) {
        R fr = R(0), fi = R(0), gr = R(0), gi = R(0);
        for (int d = 0; d < 3; d++) {
            fr += F[fidx + d].r * dirs[j][d];
            fi += F[fidx + d].i * dirs[j][d];
            if (G) {
                gr += G[fidx + d].r * dirs[j][d];
                gi += G[fidx + d].i * dirs[j][d];
            }
        }
        // psi = (F.n +- i G.n / (k c |p|)) / 2
        amp[2 * j] = a0 * R(0.5) * (fr - gsc * gi);
        amp[2 * j + 1] = a0 * R(0.5) * (fi + gsc * gr);
    }
    if (MED == FGA_MEDIUM_LAYERED) fl |= (lay << 4) | (cls << FL_ROOT_SHIFT);
}

// initial state and flags of the beam of mesh point mi and class cls
template <typename R, int MED>
__device__ __forceinline__ void beam_init_state(const ModelDev &Md, const C2<R> *__restrict__ F,
                                                const C2<R> *__restrict__ G, int nq, int np, double3 q0, double3 dq,
                                                double3 p0, double3 dp, double k, uint32_t mi, int cls, R *y, int &fl) {
    const MeshIndex x = mesh_index(nq, np, mi);
    double qd[3];
    R q[3], p[3], amp[4];
    for (int d = 0; d < 3; d++) {
        qd[d] = axis_node(q0, dq, d, x.q[d]);
        q[d] = (R)qd[d];
        p[d] = (R)axis_node(p0, dp, d, x.p[d]);
    }
    beam_amplitudes<R, MED>(Md, F, G, x.f, qd, q, p, k, cls, amp, fl);
    for (int f = 0; f < NF; f++) y[f] = R(0);
    for (int d = 0; d < 3; d++) {
        y[F_Q + d] = q[d];
        y[F_P + d] = p[d];
        y[F_DQ + 2 * (3 * d + d)] = R(1);      // dzQ = I
        y[F_DP + 2 * (3 * d + d) + 1] = R(-1); // dzP = -i I
    }
    y[F_A0] = amp[0];
    y[F_A0 + 1] = amp[1];
    y[F_A1] = amp[2];
    y[F_A1 + 1] = amp[3];
}

// |psi|^2 of a beam from its initial amplitudes (2^{3/2} psi)
template <typename R> __device__ __forceinline__ R psi_mag2(const R *a) {
    return a[0] * a[0] + a[1] * a[1] + a[2] * a[2] + a[3] * a[3];
}

// keep rule of the psi-threshold selection: |psi|^2 > eps^2 max|psi|^2 (amax2 holds the bits of the max)
template <typename R> struct MaxBits;
template <> struct MaxBits<float> {
    using U = unsigned;
    static __device__ U bits(float v) { return __float_as_uint(v); }
    static __device__ float val(U u) { return __uint_as_float(u); }
};
template <> struct MaxBits<double> {
    using U = unsigned long long;
    static __device__ U bits(double v) { return (U)__double_as_longlong(v); }
    static __device__ double val(U u) { return __longlong_as_double((long long)u); }
};

// one beam per (mesh point, requested class)
template <typename R, int MED>
__global__ void beam_init_kernel(ModelDev Md, const C2<R> *__restrict__ F, const C2<R> *__restrict__ G, int nq, int np,
                                 double3 q0, double3 dq, double3 p0, double3 dp, double k, int64_t M, int cls,
                                 int64_t off, int64_t cap, R *__restrict__ st, int32_t *__restrict__ flags,
                                 int32_t *__restrict__ ids) {
    const int64_t mi = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (mi >= M) return;
    R y[NF];
    int fl;
    beam_init_state<R, MED>(Md, F, G, nq, np, q0, dq, p0, dp, k, (uint32_t)mi, cls, y, fl);
    const int64_t b = off + mi;
    for (int f = 0; f < NF; f++) st[(int64_t)f * cap + b] = y[f];
    flags[b] = fl;
    ids[b] = (int32_t)mi;
}

// tilted layered media: the beams of [0, nb) into the layer frame x' = R x (rows of R the frame's axes):
// Q, P rotate, each row m of dzQ and dzP (the vector dQ/dz_m) rotates, S amplitudes are re-expressed in
// the S frame of the rotated P (the polarisation vector a_sv N_sv + a_sh N_sh rotates with the beam)
template <typename R>
__global__ void rotate_to_layer_frame_kernel(ModelDev Md, R *__restrict__ st, int32_t *__restrict__ flags,
                                             int64_t nb, int64_t cap) {
    const int64_t b = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (b >= nb) return;
    R y[NF];
    for (int f = 0; f < NF; f++) y[f] = st[(int64_t)f * cap + b];
    int fl = flags[b];
    rotate_state<R>(Md.R, false, true, y, fl);
    flags[b] = fl;
    for (int f = 0; f < NF; f++) st[(int64_t)f * cap + b] = y[f];
}

// The psi-threshold selection (beams with |psi| > eps max|psi|) takes three passes over the mesh, each with all
// requested classes: the largest |psi|^2, the keep masks (a byte a point) with the counts of every tile and class,
// and the initial states of the kept beams at their places in mesh order (exclusive scan of the counts, class by class).
// What bounds it: the points' transform values (24 B, 48 B with initial velocities) read twice from HBM, and
// the index and frame arithmetic of two passes.  The axis nodes come from tables in shared memory (in FP64 per point
// they took longer than the rest), the classes of a point share its loads, and the third pass lists the tile's kept
// beams first, so that whole warps form and store them.  22 M points, 13.9 M beams kept, FP32, constant medium: one launch
// per class and pass with scanned 4-byte flags 7.9 ms, this 1.9 ms (0.45 + 0.45 + 1.0).
constexpr int SEL_THREADS = 256, SEL_TILE = 1024;

struct MeshDev {
    int nq, np;
    double3 q0, dq, p0, dp;
    double k;
    uint32_t M, classes;
};

// the block's axis tables: q as Q (FP64 where the layers are decided on it), then p
template <typename R, int MED> struct MeshTable {
    using Q = typename std::conditional<MED == FGA_MEDIUM_LAYERED, double, R>::type;
    Q *q;
    R *p;
    __device__ MeshTable(const MeshDev &m, double *smem) : q(reinterpret_cast<Q *>(smem)), p(reinterpret_cast<R *>(q + 3 * m.nq)) {
        for (int i = threadIdx.x; i < 3 * m.nq; i += blockDim.x) q[i] = (Q)axis_node(m.q0, m.dq, i / m.nq, i % m.nq);
        for (int i = threadIdx.x; i < 3 * m.np; i += blockDim.x) p[i] = (R)axis_node(m.p0, m.dp, i / m.np, i % m.np);
        __syncthreads();
    }
    static size_t bytes(const MeshDev &m) { return 3 * ((size_t)m.nq * sizeof(Q) + (size_t)m.np * sizeof(R)); }
};

// |psi|^2 of the requested classes at point mi
template <typename R, int MED>
__device__ __forceinline__ void point_mags(const ModelDev &Md, const C2<R> *__restrict__ F, const C2<R> *__restrict__ G,
                                           const MeshDev &m, const MeshTable<R, MED> &tab, uint32_t mi, R *mag) {
    const MeshIndex x = mesh_index(m.nq, m.np, mi);
    double qd[3];
    R q[3], p[3];
#pragma unroll
    for (int d = 0; d < 3; d++) {
        const auto v = tab.q[d * m.nq + x.q[d]];
        qd[d] = v;
        q[d] = (R)v;
        p[d] = tab.p[d * m.np + x.p[d]];
    }
#pragma unroll
    for (int c = 0; c < 4; c++) {
        if (m.classes >> c & 1) {
            R amp[4];
            int fl;
            beam_amplitudes<R, MED>(Md, F, G, x.f, qd, q, p, m.k, c, amp, fl);
            mag[c] = psi_mag2<R>(amp);
        }
    }
}

template <typename R, int MED>
__global__ void __launch_bounds__(SEL_THREADS) psi_max_kernel(ModelDev Md, const C2<R> *__restrict__ F,
                                                              const C2<R> *__restrict__ G, MeshDev m,
                                                              typename MaxBits<R>::U *__restrict__ amax2) {
    extern __shared__ double tabs[];
    const MeshTable<R, MED> tab(m, tabs);
    R m2 = R(0);
    for (uint64_t mi = (uint64_t)blockIdx.x * SEL_THREADS + threadIdx.x; mi < m.M; mi += (uint64_t)gridDim.x * SEL_THREADS) {
        R mag[4];
        point_mags<R, MED>(Md, F, G, m, tab, (uint32_t)mi, mag);
#pragma unroll
        for (int c = 0; c < 4; c++)   // a NaN amplitude is reported by the solve, not selected on
            if ((m.classes >> c & 1) && mag[c] > m2) m2 = mag[c];
    }
    for (int o = 16; o; o >>= 1) m2 = max(m2, __shfl_xor_sync(0xffffffffu, m2, o));
    if ((threadIdx.x & 31) == 0 && m2 > R(0)) atomicMax(amax2, MaxBits<R>::bits(m2));
}

// keep[mi]: bit c set for |psi|^2 > eps2 max|psi|^2; tile_count[c][tile] and the classes' totals
template <typename R, int MED>
__global__ void __launch_bounds__(SEL_THREADS) psi_keep_kernel(ModelDev Md, const C2<R> *__restrict__ F,
                                                               const C2<R> *__restrict__ G, MeshDev m,
                                                               const typename MaxBits<R>::U *__restrict__ amax2, R eps2,
                                                               uint8_t *__restrict__ keep, uint32_t *__restrict__ tile_count,
                                                               unsigned long long *__restrict__ count) {
    extern __shared__ double tabs[];
    __shared__ unsigned n[4];
    if (threadIdx.x < 4) n[threadIdx.x] = 0;
    const MeshTable<R, MED> tab(m, tabs);
    const R lim = eps2 * MaxBits<R>::val(*amax2);
    unsigned wn[4] = {0, 0, 0, 0};
    for (int j = 0; j < SEL_TILE / SEL_THREADS; j++) {
        const uint64_t mi = (uint64_t)blockIdx.x * SEL_TILE + j * SEL_THREADS + threadIdx.x;
        unsigned kf = 0;
        if (mi < m.M) {
            R mag[4];
            point_mags<R, MED>(Md, F, G, m, tab, (uint32_t)mi, mag);
#pragma unroll
            for (int c = 0; c < 4; c++)
                if ((m.classes >> c & 1) && mag[c] > lim) kf |= 1u << c;
            keep[mi] = (uint8_t)kf;
        }
#pragma unroll
        for (int c = 0; c < 4; c++) wn[c] += __popc(__ballot_sync(0xffffffffu, kf >> c & 1));
    }
    if ((threadIdx.x & 31) == 0)
        for (int c = 0; c < 4; c++)
            if (wn[c]) atomicAdd(&n[c], wn[c]);
    __syncthreads();
    if (threadIdx.x < 4) {
        tile_count[(int64_t)threadIdx.x * gridDim.x + blockIdx.x] = n[threadIdx.x];
        if (n[threadIdx.x]) atomicAdd(&count[threadIdx.x], (unsigned long long)n[threadIdx.x]);
    }
}

// the kept beams of a tile: listed in shared memory in class and mesh order, then formed and stored
template <typename R, int MED>
__global__ void __launch_bounds__(SEL_THREADS) beam_init_kept_kernel(ModelDev Md, const C2<R> *__restrict__ F,
                                                                     const C2<R> *__restrict__ G, MeshDev m,
                                                                     const uint8_t *__restrict__ keep,
                                                                     const uint32_t *__restrict__ tile_off, int64_t cap,
                                                                     R *__restrict__ st, int32_t *__restrict__ flags,
                                                                     int32_t *__restrict__ ids) {
    constexpr int NW = SEL_THREADS / 32, PER = SEL_TILE / SEL_THREADS;
    __shared__ uint16_t list[4 * SEL_TILE];       // class << 10 | point of the tile
    __shared__ unsigned cnt[4 * NW], first[4 * NW + 1];
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint64_t tile0 = (uint64_t)blockIdx.x * SEL_TILE;
    unsigned bal[PER][4], n[4] = {0, 0, 0, 0};
#pragma unroll
    for (int j = 0; j < PER; j++) {   // a warp's points are consecutive
        const uint64_t mi = tile0 + (w * PER + j) * 32 + lane;
        const unsigned kf = mi < m.M ? keep[mi] : 0u;
#pragma unroll
        for (int c = 0; c < 4; c++) {
            bal[j][c] = __ballot_sync(0xffffffffu, kf >> c & 1);
            n[c] += __popc(bal[j][c]);
        }
    }
    if (lane == 0)
        for (int c = 0; c < 4; c++) cnt[c * NW + w] = n[c];
    __syncthreads();
    if (threadIdx.x == 0) {
        unsigned t = 0;
        for (int i = 0; i < 4 * NW; i++) {
            first[i] = t;
            t += cnt[i];
        }
        first[4 * NW] = t;
    }
    __syncthreads();
#pragma unroll
    for (int c = 0; c < 4; c++) {
        unsigned at = first[c * NW + w];
#pragma unroll
        for (int j = 0; j < PER; j++) {
            if (bal[j][c] >> lane & 1)
                list[at + __popc(bal[j][c] & ((1u << lane) - 1))] = (uint16_t)(c << 10 | ((w * PER + j) * 32 + lane));
            at += __popc(bal[j][c]);
        }
    }
    __syncthreads();
    for (unsigned i = threadIdx.x; i < first[4 * NW]; i += SEL_THREADS) {
        const int c = list[i] >> 10;
        const uint32_t mi = (uint32_t)tile0 + (list[i] & (SEL_TILE - 1));
        R y[NF];
        int fl;
        beam_init_state<R, MED>(Md, F, G, m.nq, m.np, m.q0, m.dq, m.p0, m.dp, m.k, mi, c, y, fl);
        const int64_t b = (int64_t)tile_off[(int64_t)c * gridDim.x + blockIdx.x] + (i - first[c * NW]);
        for (int f = 0; f < NF; f++) st[(int64_t)f * cap + b] = y[f];
        flags[b] = fl;
        ids[b] = (int32_t)mi;
    }
}

// F (and G from g, if both are given) = the transform of Eq. psi in the per-axis pair layout
// [a0][a1][a2][3], a_d = iq_d * np + jp_d.  Synchronises s before its temporaries are released; reports
// a tensor-core wait that ran out as FGA_ERR_TIMEOUT.
template <typename R>
static fga_status transform_typed(const fga_init_desc *d, const double2 *f, const double2 *g, C2<R> *F, C2<R> *G,
                                  cudaStream_t s) {
    const int A = d->nq * d->np;
    ScopedDevBuf Kb, T1, T2, tsb;
    FGA_TRY(T1.ensure(sizeof(C2<R>) * (size_t)d->ny[0] * d->ny[1] * A * 3));
    FGA_TRY(T2.ensure(sizeof(C2<R>) * (size_t)d->ny[0] * A * A * 3));
    FGA_TRY(tsb.ensure(64));
    TransformScratch ts;
    ts.amax = tsb.as<float>();
    ts.err = reinterpret_cast<int *>(tsb.as<char>() + 16);
    FGA_CUDA(cudaMemsetAsync(tsb.p, 0, 64, s));
    if constexpr (sizeof(R) == 4) {
        KernelMatrices K;
        K.nq = d->nq;
        K.np = d->np;
        K.k = d->k;
        size_t total = 0;
        for (int a = 0; a < 3; a++) {
            KernelMatrix &X = K.ax[a];
            tc_kernel_shape(A, d->ny[a], X);
            X.q0 = d->q0[a];
            X.dq = d->dq[a];
            X.p0 = d->p0[a];
            X.dp = d->dp[a];
            X.y0 = d->y0[a];
            X.dy = d->dy[a];
            total += X.bytes;
            ts.S[a] = kernel_row_sum_max(d->nq, d->q0[a], d->dq[a], d->ny[a], d->y0[a], d->dy[a], d->k);
        }
        FGA_TRY(Kb.ensure(total));
        unsigned char *at = Kb.as<unsigned char>();
        for (int a = 0; a < 3; a++) {
            K.ax[a].B = at;
            at += K.ax[a].bytes;
        }
        FGA_TRY(tc_kernel_matrices(K, s));
        float2 *t1 = T1.as<float2>(), *t2 = T2.as<float2>();
        FGA_TRY(fbi_transform_f32(d, f, K, t1, t2, reinterpret_cast<float2 *>(F), ts, s));
        if (g && G) FGA_TRY(fbi_transform_f32(d, g, K, t1, t2, reinterpret_cast<float2 *>(G), ts, s));
    } else {
        FGA_TRY(Kb.ensure(sizeof(C2<R>) * (size_t)A * (d->ny[0] + d->ny[1] + d->ny[2])));
        C2<R> *Kax[3];
        Kax[0] = Kb.as<C2<R>>();
        Kax[1] = Kax[0] + (size_t)A * d->ny[0];
        Kax[2] = Kax[1] + (size_t)A * d->ny[1];
        for (int ax = 0; ax < 3; ax++) {
            const int tot = A * d->ny[ax];
            ProfScope ps(P_DECOMP, s);
            fbi_axis_kernel<R><<<(tot + 255) / 256, 256, 0, s>>>(Kax[ax], d->nq, d->np, d->ny[ax], d->q0[ax], d->dq[ax],
                                                                d->p0[ax], d->dp[ax], d->y0[ax], d->dy[ax], d->k);
        }
        FGA_CUDA(cudaGetLastError());
        FGA_TRY(fbi_transform_f64(d, f, Kax, T1.as<C2<R>>(), T2.as<C2<R>>(), F, s));
        if (g && G) FGA_TRY(fbi_transform_f64(d, g, Kax, T1.as<C2<R>>(), T2.as<C2<R>>(), G, s));
    }
    // the temporaries are released when this scope ends; make sure the stream is done with them
    int terr = 0;
    if (sizeof(R) == 4) FGA_CUDA(cudaMemcpyAsync(&terr, ts.err, sizeof terr, cudaMemcpyDeviceToHost, s));
    FGA_CUDA(cudaStreamSynchronize(s));
    if (sizeof(R) == 4) {
        if (terr) {
            set_error("wave-packet transform: a tensor-core wait ran out");
            return FGA_ERR_TIMEOUT;
        }
    }
    return FGA_OK;
}

// Beam-set storage for the class counts in b->n_cls: class blocks in class order, capacity rounded
// to 32 (layered media: growth x the initial count, for the children created at interfaces)
static fga_status beams_allocate(fga_beams *b, const fga_init_desc *d, cudaStream_t s) {
    int64_t off = 0;
    for (int c = 0; c < 4; c++) {
        b->off_cls[c] = off;
        off += b->n_cls[c];
    }
    b->nb = off;
    if (b->layered) {
        const double growth = d->growth > 0 ? std::max(1.0, d->growth) : 4.0;
        b->cap = ((int64_t)std::ceil(growth * (double)off) + 31) / 32 * 32;
    } else {
        b->cap = (off + 31) / 32 * 32;
    }
    b->cap = std::max<int64_t>(b->cap, 32);
    const size_t rb = d->precision == FGA_PREC_FP64 ? 8 : 4;
    FGA_TRY(b->state.ensure(rb * NFS * b->cap));
    // the Q compensation starts at zero
    FGA_CUDA(cudaMemsetAsync(static_cast<char *>(b->state.p) + rb * F_QC * b->cap, 0, rb * 3 * b->cap, s));
    FGA_TRY(b->flags.ensure(4 * b->cap));
    FGA_TRY(b->id.ensure(4 * b->cap));
    if (b->layered) {
        FGA_TRY(b->path.ensure(8 * b->cap));
        FGA_TRY(b->counts.ensure(16));
        const unsigned long long c0[2] = {(unsigned long long)off, 0ull};
        FGA_CUDA(cudaMemsetAsync(b->path.p, 0, 8 * b->cap, s));
        FGA_CUDA(cudaMemcpyAsync(b->counts.p, c0, sizeof c0, cudaMemcpyHostToDevice, s));
        FGA_CUDA(cudaStreamSynchronize(s));
    }
    return FGA_OK;
}

template <typename R, int MED>
static fga_status decompose_medium(const fga_model *m, const fga_init_desc *d, fga_beams *b, const C2<R> *F,
                                   const C2<R> *G, cudaStream_t s) {
    const int64_t M = (int64_t)d->nq * d->nq * d->nq * d->np * d->np * d->np;
    const double3 q0 = {d->q0[0], d->q0[1], d->q0[2]}, dq = {d->dq[0], d->dq[1], d->dq[2]};
    const double3 p0 = {d->p0[0], d->p0[1], d->p0[2]}, dp = {d->dp[0], d->dp[1], d->dp[2]};
    const bool select = d->psi_rel_min > 0;
    using U = typename MaxBits<R>::U;
    ScopedDevBuf keepb, tileb, selb;
    const MeshDev mesh = {d->nq, d->np, q0, dq, p0, dp, d->k, (uint32_t)M, d->class_mask};
    const unsigned tiles = (unsigned)((M + SEL_TILE - 1) / SEL_TILE);
    if (select) {
        // Step 1 of Fig. fig:FGA_alg chooses the beams worth propagating: |psi| > eps max|psi|, the maximum
        // over every requested class and mesh point
        using U = typename MaxBits<R>::U;
        const R eps2 = (R)(d->psi_rel_min * d->psi_rel_min);
        const size_t smem = MeshTable<R, MED>::bytes(mesh);
        FGA_TRY(selb.ensure(64));
        U *amax2 = selb.as<U>();
        unsigned long long *cnt = reinterpret_cast<unsigned long long *>(selb.as<char>() + 16);
        FGA_CUDA(cudaMemsetAsync(selb.p, 0, 64, s));
        FGA_TRY(keepb.ensure((size_t)M));
        FGA_TRY(tileb.ensure(sizeof(uint32_t) * 4 * (size_t)tiles));
        {
            ProfScope ps(P_DECOMP, s);
            psi_max_kernel<R, MED><<<std::min(tiles, 152u * 8u), SEL_THREADS, smem, s>>>(m->dev, F, G, mesh, amax2);
        }
        FGA_CUDA(cudaGetLastError());
        {
            ProfScope ps(P_DECOMP, s);
            psi_keep_kernel<R, MED><<<tiles, SEL_THREADS, smem, s>>>(m->dev, F, G, mesh, amax2, eps2, keepb.as<uint8_t>(),
                                                                     tileb.as<uint32_t>(), cnt);
        }
        FGA_CUDA(cudaGetLastError());
        unsigned long long hc[4];
        FGA_CUDA(cudaMemcpyAsync(hc, cnt, sizeof hc, cudaMemcpyDeviceToHost, s));
        FGA_CUDA(cudaStreamSynchronize(s));
        int64_t tot = 0;
        for (int c = 0; c < 4; c++) {
            b->n_cls[c] = (int64_t)hc[c];
            tot += b->n_cls[c];
        }
        FGA_CHECK(tot < (int64_t)1 << 31, "fga_decompose: more than 2^31 selected beams");
    } else {
        for (int c = 0; c < 4; c++) b->n_cls[c] = (d->class_mask & (1u << c)) ? M : 0;
    }
    FGA_TRY(beams_allocate(b, d, s));
    if (select && b->nb > 0) {
        FGA_TRY(scan_exclusive_u32(tileb.as<uint32_t>(), 4 * (int64_t)tiles, s));
        ProfScope ps(P_DECOMP, s);
        beam_init_kept_kernel<R, MED><<<tiles, SEL_THREADS, 0, s>>>(m->dev, F, G, mesh, keepb.as<uint8_t>(),
                                                                    tileb.as<uint32_t>(), b->cap, b->state.as<R>(),
                                                                    b->flags.as<int32_t>(), b->id.as<int32_t>());
        FGA_CUDA(cudaGetLastError());
    }
    for (int cls = 0; cls < 4 && !select; cls++) {
        if (!b->n_cls[cls]) continue;
        ProfScope ps(P_DECOMP, s);
        beam_init_kernel<R, MED><<<(unsigned)((M + 127) / 128), 128, 0, s>>>(
            m->dev, F, G, d->nq, d->np, q0, dq, p0, dp, d->k, M, cls, b->off_cls[cls], b->cap, b->state.as<R>(),
            b->flags.as<int32_t>(), b->id.as<int32_t>());
        FGA_CUDA(cudaGetLastError());
    }
    if (MED == FGA_MEDIUM_LAYERED && m->dev.tilted) {
        b->tilted = true;
        for (int i = 0; i < 9; i++) b->R[i] = m->dev.R[i];
        if (b->nb > 0) {
            ProfScope ps(P_DECOMP, s);
            rotate_to_layer_frame_kernel<R><<<(unsigned)((b->nb + 127) / 128), 128, 0, s>>>(
                m->dev, b->state.as<R>(), b->flags.as<int32_t>(), b->nb, b->cap);
        }
        FGA_CUDA(cudaGetLastError());
    }
    // the selection scratch is released when this scope ends
    FGA_CUDA(cudaStreamSynchronize(s));
    return FGA_OK;
}

template <typename R>
static fga_status decompose_typed(const fga_model *m, const fga_init_desc *d, fga_beams *b, cudaStream_t s) {
    const int A = d->nq * d->np;
    ScopedDevBuf Fb, Gb;
    const size_t Fn = (size_t)A * A * A * 3;
    FGA_TRY(Fb.ensure(sizeof(C2<R>) * Fn));
    const C2<R> *G = nullptr;
    if (d->g) {
        FGA_TRY(Gb.ensure(sizeof(C2<R>) * Fn));
        G = Gb.as<C2<R>>();
    }
    FGA_TRY(transform_typed<R>(d, static_cast<const double2 *>(d->f), static_cast<const double2 *>(d->g),
                               Fb.as<C2<R>>(), Gb.as<C2<R>>(), s));
    const C2<R> *F = Fb.as<C2<R>>();
    switch (m->dev.kind) {
    case FGA_MEDIUM_CONST: FGA_TRY((decompose_medium<R, FGA_MEDIUM_CONST>(m, d, b, F, G, s))); break;
    case FGA_MEDIUM_SINE: FGA_TRY((decompose_medium<R, FGA_MEDIUM_SINE>(m, d, b, F, G, s))); break;
    case FGA_MEDIUM_GRID: FGA_TRY((decompose_medium<R, FGA_MEDIUM_GRID>(m, d, b, F, G, s))); break;
    default: FGA_TRY((decompose_medium<R, FGA_MEDIUM_LAYERED>(m, d, b, F, G, s))); break;
    }
    // F and G are released when this scope ends; make sure the stream is done with them
    FGA_CUDA(cudaStreamSynchronize(s));
    return FGA_OK;
}

fga_status decompose_impl(const fga_model *m, const fga_init_desc *d, fga_beams **out, cudaStream_t s) {
    FGA_CHECK(m && d && out, "fga_decompose: NULL argument");
    FGA_CHECK(std::isfinite(d->k) && d->k > 0, "fga_decompose: k must be > 0");
    FGA_CHECK(d->f != nullptr, "fga_decompose: f is NULL");
    FGA_CHECK(d->nq >= 1 && d->np >= 1, "fga_decompose: nq, np must be >= 1");
    FGA_CHECK(d->ny[0] >= 1 && d->ny[1] >= 1 && d->ny[2] >= 1, "fga_decompose: ny must be >= 1");
    FGA_CHECK((d->class_mask & 15u) != 0 && (d->class_mask & ~15u) == 0, "fga_decompose: class_mask must be in 1..15");
    FGA_CHECK(d->precision == FGA_PREC_FP32 || d->precision == FGA_PREC_FP64, "fga_decompose: bad precision");
    FGA_CHECK(std::isfinite(d->psi_rel_min) && d->psi_rel_min >= 0 && d->psi_rel_min < 1,
              "fga_decompose: psi_rel_min must be in [0, 1)");
    for (int a = 0; a < 3; a++) FGA_CHECK(d->dy[a] > 0 && d->dq[a] > 0 && d->dp[a] > 0, "fga_decompose: spacings must be > 0");
    const int64_t M = (int64_t)d->nq * d->nq * d->nq * d->np * d->np * d->np;
    // mesh indices are int32; without a selection every mesh point of every class is a beam slot
    FGA_CHECK(M < (int64_t)1 << 31, "fga_decompose: more than 2^31 mesh points");
    if (!(d->psi_rel_min > 0)) {
        int nc = 0;
        for (int c = 0; c < 4; c++) nc += (d->class_mask >> c) & 1;
        FGA_CHECK(M * nc < (int64_t)1 << 31, "fga_decompose: more than 2^31 beams");
    }
    fga_beams *b = new fga_beams();
    b->precision = d->precision;
    b->k = d->k;
    double vol = 1.0;
    for (int a = 0; a < 3; a++) vol *= d->dq[a] * d->dp[a];
    b->w = vol / std::pow(2.0 * M_PI / d->k, 4.5);
    b->layered = m->dev.kind == FGA_MEDIUM_LAYERED;
    if (b->layered) {
        b->gmax = d->max_interfaces > 0 ? d->max_interfaces : 4;
        b->rel_min = d->child_rel_min > 0 ? d->child_rel_min : 1e-6;
    }
    const fga_status st =
        d->precision == FGA_PREC_FP64 ? decompose_typed<double>(m, d, b, s) : decompose_typed<float>(m, d, b, s);
    if (st != FGA_OK) {
        fga_beams_destroy(b);
        return st;
    }
    b->last_stream = s;
    *out = b;
    return FGA_OK;
}

fga_status transform_impl(const fga_init_desc *d, void *F_out, cudaStream_t s) {
    FGA_CHECK(d && F_out, "fga_transform: NULL argument");
    FGA_CHECK(std::isfinite(d->k) && d->k > 0, "fga_transform: k must be > 0");
    FGA_CHECK(d->f != nullptr, "fga_transform: f is NULL");
    FGA_CHECK(d->nq >= 1 && d->np >= 1, "fga_transform: nq, np must be >= 1");
    FGA_CHECK(d->ny[0] >= 1 && d->ny[1] >= 1 && d->ny[2] >= 1, "fga_transform: ny must be >= 1");
    FGA_CHECK(d->precision == FGA_PREC_FP32 || d->precision == FGA_PREC_FP64, "fga_transform: bad precision");
    for (int a = 0; a < 3; a++) FGA_CHECK(d->dy[a] > 0 && d->dq[a] > 0 && d->dp[a] > 0, "fga_transform: spacings must be > 0");
    const int64_t A = (int64_t)d->nq * d->np;
    FGA_CHECK(A * A * A * 3 < (int64_t)1 << 31, "fga_transform: more than 2^31 output values");
    if (d->precision == FGA_PREC_FP64)
        return transform_typed<double>(d, static_cast<const double2 *>(d->f), nullptr, static_cast<C2<double> *>(F_out),
                                       nullptr, s);
    return transform_typed<float>(d, static_cast<const double2 *>(d->f), nullptr, static_cast<C2<float> *>(F_out),
                                  nullptr, s);
}

}  // namespace fga
