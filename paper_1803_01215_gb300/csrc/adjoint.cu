// Reverse sweep through the PDHG iterations (the adjoint of Algorithm 1 run for
// exactly K iterations), with the iterates checkpointed every C iterations.
//
// For a point solved in K iterations, V_K = fval(x^K, p^K) (Algorithm 1's value
// at the final iterate) is a smooth function of the cost weights W, the centre
// c, the dynamics parameters and the query point x (through x_N = x and the
// initial guess x^0 = x + r u).  This kernel returns its exact gradient by
// reverse-mode differentiation of the K iterations:
//   forward   run the K iterations again from the counter-based initial guess,
//             storing (x, p, z) at iterations 0, C, 2C, ... in workspace;
//   backward  segment by segment, newest first: the segment's C iterations are run
//             once more from its checkpoint, each leaving what its transpose
//             needs in a history buffer, and then for k = last .. first the
//             transposed Jacobian of step k is applied to the adjoint (xbar, pbar,
//             zbar), accumulating parameter adjoints.  2 K forward and K
//             transposed steps per point.  The history holds S = C steps up to
//             C = 64; a longer segment is run once with checkpoints every S steps
//             and then by these, as a segment is by its own: 3 K forward steps, and
//             the workspace stays the K / C checkpoints that were asked for, C / S
//             more and S steps.
// At a converged point this equals the envelope gradient of hj_solve_grad.
// One CTA of G warps per point (lane l <-> node l + 1; lanes 0..D-1 also hold one
// coordinate each of node 0); neighbour terms go through per-lane shared-memory
// slots, as in the solver, two barriers per step.  The history of step k - 1 is
// copied to shared memory by cp.async while step k is transposed.
// Families: quadratic (d <= 4) and quadcopter (d = 12).
//
// What bounds it: instruction issue at 8 warps per SM (255 registers; about 1100
// instructions per warp and iteration, 2 forward steps and a transposed one).
// Rebuilding s^k from its checkpoint for every k cost K C / 2 forward steps; with the
// history a segment is run once, in 64 bytes per lane and step that mostly stay in
// L2.  An FP64 instruction holds this GPU's FP64 pipe about 64 cycles per warp: the
// parameter sums of FP32 iterates are therefore three floats per lane (StepSum), the
// constant factors are applied once per point, and node 0's sums run on the lane that
// owns the coordinate.  Measured through the autograd call (quadcopter, 2048 points,
// N = 64, 1330 iterations on average, C = 32): 86.5 -> 13.4 ms, of which the history
// took 69 ms, its 64-byte chunk-major layout (from 96 bytes, lane-major) 2 ms and the
// FP32-pipe sums 2 ms.  Register caps of 168 and 128 (12 and 16 warps per SM, 0.2 and
// 0.6 KB of spills) ran 17 and 20 ms; segments of 8 and 16 steps 21 and 19 ms against 18.
#include <cuda_runtime.h>

#include "families.cuh"
#include "hj_internal.cuh"
#include "hjpdhg.h"
#include "warp_solver.cuh"

namespace hj {

namespace {

// ---------------------------------------------------------------- per-node family math
// Quadcopter pieces in the iterate type (the solver's formulas, written out
// with their intermediates so the reverse rules can reuse them).
template <typename T>
struct QCNode {
  T a[3], J[9], H2[27];   // thrust direction, d a / d angles, second derivatives
};

template <typename T>
__device__ __forceinline__ void qc_node(const T (&x)[12], QCNode<T>& n) {
  T sps, cps, sth, cth, sph, cph;
  sin_cos<T>(x[3], &sps, &cps);
  sin_cos<T>(x[4], &sth, &cth);
  sin_cos<T>(x[5], &sph, &cph);
  n.a[0] = sph * sps + cph * cps * sth;
  n.a[1] = -cps * sph + cph * sth * sps;
  n.a[2] = cth * cph;
  // J[3r + c] = d a_r / d angle_c, angles (psi, theta, phi)
  n.J[0] = sph * cps - cph * sps * sth; n.J[1] = cph * cps * cth; n.J[2] = cph * sps - sph * cps * sth;
  n.J[3] = sps * sph + cph * sth * cps; n.J[4] = cph * cth * sps; n.J[5] = -cps * cph - sph * sth * sps;
  n.J[6] = T(0);                        n.J[7] = -sth * cph;       n.J[8] = -cth * sph;
  // H2[9r + 3c + k] = d^2 a_r / d angle_c d angle_k
  T* h = n.H2;
  // a0
  h[0] = -n.a[0];                 h[1] = -cph * sps * cth;        h[2] = cph * cps + sph * sps * sth;
  h[3] = h[1];                    h[4] = -cph * cps * sth;        h[5] = -sph * cps * cth;
  h[6] = h[2];                    h[7] = h[5];                    h[8] = -n.a[0];
  // a1
  h[9] = -n.a[1];                 h[10] = cph * cth * cps;        h[11] = sps * cph - sph * sth * cps;
  h[12] = h[10];                  h[13] = -cph * sth * sps;       h[14] = -sph * cth * sps;
  h[15] = h[11];                  h[16] = h[14];                  h[17] = -n.a[1];
  // a2
  h[18] = T(0); h[19] = T(0); h[20] = T(0);
  h[21] = T(0); h[22] = -n.a[2];  h[23] = sth * sph;
  h[24] = T(0); h[25] = h[23];    h[26] = -n.a[2];
}

struct QCPar { double m, ah, gz, eps; };

// p' = prox(x, v) of the quadcopter H (Sherman-Morrison on rows 6-8)
template <typename T>
__device__ __forceinline__ void qc_prox(const QCNode<T>& n, const QCPar& q, T L, const T (&x)[12],
                                        const T (&v)[12], T (&pp)[12]) {
  const T al = T(1) + L * T(q.eps), ial = T(1) / al, irate = T(1) / (al + L), minv = T(1.0 / q.m);
  for (int k = 0; k < 6; ++k) pp[k] = (v[k] - L * x[6 + k]) * ial;
  for (int k = 9; k < 12; ++k) pp[k] = v[k] * irate;
  T w[3], b[3];
  for (int r = 0; r < 3; ++r) {
    w[r] = v[6 + r] - L * (T(q.ah) * n.a[r] - (r == 2 ? T(q.gz) : T(0)));
    b[r] = n.a[r] * minv;
  }
  const T bb = b[0] * b[0] + b[1] * b[1] + b[2] * b[2];
  const T bw = b[0] * w[0] + b[1] * w[1] + b[2] * w[2];
  const T f = L * bw / (al + L * bb);
  for (int r = 0; r < 3; ++r) pp[6 + r] = (w[r] - f * b[r]) * ial;
}

// grad_x H(x, p) of the quadcopter
template <typename T>
__device__ __forceinline__ void qc_gradx(const QCNode<T>& n, const QCPar& q, const T (&p)[12],
                                         T (&g)[12]) {
  const T minv = T(1.0 / q.m);
  const T s = n.a[0] * p[6] + n.a[1] * p[7] + n.a[2] * p[8];
  const T coef = T(q.ah) + s * minv * minv;
  g[0] = g[1] = g[2] = T(0);
  for (int c = 0; c < 3; ++c) g[3 + c] = coef * (n.J[c] * p[6] + n.J[3 + c] * p[7] + n.J[6 + c] * p[8]);
  for (int k = 0; k < 3; ++k) { g[6 + k] = p[k]; g[9 + k] = p[3 + k]; }
}

// grad_p H(x, p) = f0 + B B^T p + eps p
template <typename T>
__device__ __forceinline__ void qc_gradp(const QCNode<T>& n, const QCPar& q, const T (&x)[12],
                                         const T (&p)[12], T (&g)[12]) {
  const T minv = T(1.0 / q.m), e = T(q.eps);
  const T u0 = (n.a[0] * p[6] + n.a[1] * p[7] + n.a[2] * p[8]) * minv;
  for (int k = 0; k < 3; ++k) { g[k] = x[6 + k] + e * p[k]; g[3 + k] = x[9 + k] + e * p[3 + k]; }
  for (int r = 0; r < 3; ++r)
    g[6 + r] = T(q.ah) * n.a[r] - (r == 2 ? T(q.gz) : T(0)) + n.a[r] * minv * u0 + e * p[6 + r];
  for (int k = 9; k < 12; ++k) g[k] = p[k] + e * p[k];
}

// d H / d (m, a_h, g_z, eps) at (x, p)
template <typename T>
__device__ __forceinline__ void qc_dHdpar(const QCNode<T>& n, const QCPar& q, const T (&p)[12],
                                          double (&o)[4]) {
  const double s = (double)(n.a[0] * p[6] + n.a[1] * p[7] + n.a[2] * p[8]);
  double pp = 0.0;
  for (int k = 0; k < 12; ++k) pp += (double)p[k] * (double)p[k];
  o[0] = -s * s / (q.m * q.m * q.m);
  o[1] = s;
  o[2] = -(double)p[8];
  o[3] = 0.5 * pp;
}

// A sum over iterations.  FP64 terms are added in FP64.  FP32 terms are added into
// three floats by Knuth's error-free TwoSum (the rounding error of the first sum
// goes into the second, the second's into the third), which is folded into an FP64
// sum after 64 steps at most: within 64 steps of 4 terms (a_h) the three floats hold the
// sum to 256^3 2^-72 of it, under the 256 2^-53 that adding the converted terms in FP64
// would give, and every instruction runs on the FP32 pipe.  The callers add only terms
// below 2^118 this way, so that no sum of 256 overflows, and larger ones to FP64 (wide).
template <typename T>
struct StepSum {
  double s = 0.0;
  __device__ __forceinline__ void add(double t) { s += t; }
  __device__ __forceinline__ double take() { const double r = s; s = 0.0; return r; }
};
template <>
struct StepSum<float> {
  float a = 0.f, b = 0.f, c = 0.f;
  __device__ __forceinline__ static float two_sum(float& h, float t) {
    const float n = __fadd_rn(h, t), bb = __fsub_rn(n, h);
    const float e = __fadd_rn(__fsub_rn(h, __fsub_rn(n, bb)), __fsub_rn(t, bb));
    h = n;
    return e;
  }
  __device__ __forceinline__ void add(float t) { c = __fadd_rn(c, two_sum(b, two_sum(a, t))); }
  __device__ __forceinline__ double take() {
    const double r = (double)a + ((double)b + (double)c);
    a = b = c = 0.f;
    return r;
  }
};

// Whether one of the terms is too large for a StepSum (a NaN is not: it stays one there).
template <typename... U>
__device__ __forceinline__ bool wide(float t, U... ts) {
  float m = fabsf(t);
  ((m = fmaxf(m, fabsf(ts))), ...);
  return m >= 0x1p118f;
}
template <typename... U>
__device__ __forceinline__ bool wide(double, U...) { return false; }

// Sums over the iterations that the parameter adjoints are linear in; the constant
// factors are applied once per point (qc_par).
// big: the lane's FP64 sums.
template <typename T>
struct QCStep { StepSum<T> ma, mc, ah, gz, eps; };
struct QCSums { double ma, mc, ah, gz, eps; };
__device__ __forceinline__ void qc_par(const QCSums& s, const QCPar& q, double (&par)[4]) {
  par[0] += -s.ma / (q.m * q.m) - 2.0 * s.mc / (q.m * q.m * q.m);
  par[1] += s.ah;
  par[2] += s.gz;
  par[3] += s.eps;
}

// Reverse of qc_prox: given pb = dL/dp', add dL/dv to vb, dL/dx to xb (rows
// 6-11 and angles), the sums of dL/d(m, a_h, g_z, eps) to par.
template <typename T>
__device__ __forceinline__ void qc_prox_vjp(const QCNode<T>& n, const QCPar& q, T L,
                                            const T (&v)[12], const T (&pp)[12],
                                            const T (&pb)[12], T (&vb)[12], T (&xb)[12],
                                            QCStep<T>& par, QCSums& big) {
  const T al = T(1) + L * T(q.eps), ial = T(1) / al, irate = T(1) / (al + L);
  const T m = T(q.m), minv = T(1) / m;
  T alb = T(0);
  for (int k = 0; k < 6; ++k) {
    vb[k] += pb[k] * ial;
    xb[6 + k] += -L * ial * pb[k];
    alb += -pb[k] * pp[k] * ial;
  }
  for (int k = 9; k < 12; ++k) {
    vb[k] += pb[k] * irate;
    alb += -pb[k] * pp[k] * irate;               // d/d(al) of v/(al + L)
  }
  T w[3], b[3];
  for (int r = 0; r < 3; ++r) {
    w[r] = v[6 + r] - L * (T(q.ah) * n.a[r] - (r == 2 ? T(q.gz) : T(0)));
    b[r] = n.a[r] * minv;
  }
  const T bb = b[0] * b[0] + b[1] * b[1] + b[2] * b[2];
  const T bw = b[0] * w[0] + b[1] * w[1] + b[2] * w[2];
  const T den = al + L * bb;
  const T f = L * bw / den;
  T wb[3], bbar[3], fb = T(0);
  for (int r = 0; r < 3; ++r) {
    wb[r] = pb[6 + r] * ial;
    fb += -pb[6 + r] * b[r] * ial;
    bbar[r] = -f * pb[6 + r] * ial;
    alb += -pb[6 + r] * pp[6 + r] * ial;
  }
  const T bwb = fb * L / den;
  const T denb = -fb * f / den;
  alb += denb;
  const T bbb = L * denb;
  for (int r = 0; r < 3; ++r) {
    bbar[r] += bwb * w[r] + T(2) * bbb * b[r];
    wb[r] += bwb * b[r];
  }
  T ab[3], tm[3], ta[3];
  for (int r = 0; r < 3; ++r) {
    ab[r] = bbar[r] * minv;
    tm[r] = bbar[r] * n.a[r];
    vb[6 + r] += wb[r];
    ab[r] += -L * T(q.ah) * wb[r];
    ta[r] = -(L * wb[r] * n.a[r]);
  }
  const T tg = L * wb[2], te = L * alb;           // al = 1 + L eps
  if (!wide(tm[0], tm[1], tm[2], ta[0], ta[1], ta[2], tg, te)) {
    for (int r = 0; r < 3; ++r) { par.ma.add(tm[r]); par.ah.add(ta[r]); }
    par.gz.add(tg);
    par.eps.add(te);
  } else {
    for (int r = 0; r < 3; ++r) { big.ma += (double)tm[r]; big.ah += (double)ta[r]; }
    big.gz += (double)tg;
    big.eps += (double)te;
  }
  for (int c = 0; c < 3; ++c)
    xb[3 + c] += n.J[c] * ab[0] + n.J[3 + c] * ab[1] + n.J[6 + c] * ab[2];
}

// Reverse of qc_gradx: given gb = dL/dg, add dL/dx (angles) to xb, dL/dp to pb,
// the sums of dL/d(m, a_h) to par.
template <typename T>
__device__ __forceinline__ void qc_gradx_vjp(const QCNode<T>& n, const QCPar& q, const T (&p)[12],
                                             const T (&gb)[12], T (&xb)[12], T (&pb)[12],
                                             QCStep<T>& par, QCSums& big) {
  const T minv = T(1.0 / q.m);
  for (int k = 0; k < 3; ++k) { pb[k] += gb[6 + k]; pb[3 + k] += gb[9 + k]; }
  T qv[3] = {p[6], p[7], p[8]};
  const T s = n.a[0] * qv[0] + n.a[1] * qv[1] + n.a[2] * qv[2];
  const T coef = T(q.ah) + s * minv * minv;
  T h[3], hb[3], coefb = T(0);
  for (int c = 0; c < 3; ++c) {
    h[c] = n.J[c] * qv[0] + n.J[3 + c] * qv[1] + n.J[6 + c] * qv[2];
    coefb += gb[3 + c] * h[c];
    hb[c] = coef * gb[3 + c];
  }
  T qb[3], Jb[9];
  for (int r = 0; r < 3; ++r) {
    qb[r] = n.J[3 * r] * hb[0] + n.J[3 * r + 1] * hb[1] + n.J[3 * r + 2] * hb[2];
    for (int c = 0; c < 3; ++c) Jb[3 * r + c] = qv[r] * hb[c];
  }
  const T sb = coefb * minv * minv, tc = s * coefb;
  if (!wide(coefb, tc)) {
    par.ah.add(coefb);
    par.mc.add(tc);
  } else {
    big.ah += (double)coefb;
    big.mc += (double)tc;
  }
  T ab[3];
  for (int r = 0; r < 3; ++r) { ab[r] = sb * qv[r]; qb[r] += sb * n.a[r]; }
  for (int r = 0; r < 3; ++r) pb[6 + r] += qb[r];
  for (int k = 0; k < 3; ++k) {
    T acc = n.J[k] * ab[0] + n.J[3 + k] * ab[1] + n.J[6 + k] * ab[2];
    for (int r = 0; r < 3; ++r)
      for (int c = 0; c < 3; ++c) acc += Jb[3 * r + c] * n.H2[9 * r + 3 * c + k];
    xb[3 + k] += acc;
  }
}

constexpr int kHistSteps = 64;   // steps whose history is kept, and which a StepSum adds, at most

// 16-byte asynchronous copy global -> shared (a thread's own data: no barrier)
__device__ __forceinline__ void cp_async16(void* dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;"
               ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int n>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(n) : "memory"); }

// A lane's history of one step (quadcopter; the quadratic family's transposed step
// needs none): the angles of x^k, v_{6..8}, and the rows of p^{k+1} that are linear
// in v and x alone, 16 values = 64 bytes (FP32) per lane, kept as 16-byte chunks,
// chunk-major over the lanes so that a warp's accesses are contiguous.
template <int FAM>
constexpr int hist_vals() { return FAM == 1 ? 16 : 0; }
template <typename T, int FAM>
constexpr int hist_chunks() { return hist_vals<FAM>() * (int)sizeof(T) / 16; }

template <typename T, int FAM, int D, int G>
struct AdjShared {
  static constexpr int DP = padded_dim<T, D>();
  alignas(16) T zs[32 * G][DP];
  alignas(16) T ps[32 * G][DP];
  alignas(16) T node0[DP];                       // z_0 (forward), x0bar' ginv (backward)
  alignas(16) T hist[2][32 * G][FAM == 1 ? 16 : 1];
  QCSums sums[FAM == 1 ? 32 * G : 1];
  double red[G][D + 4];
  double vpar[G][4];                             // the value's own part of the parameter adjoints
  double c[D], W0[D], c0[D];                     // node 0: the centre; the value's part of Wbar, cbar
  unsigned long long item;
};

// FAM 0: quadratic (H = |p|^2 / 2), 1: quadcopter
template <typename T, int FAM, int D, int G>
__global__ void __launch_bounds__(32 * G) adjoint_kernel(const AdjArgs<T> a) {
  extern __shared__ __align__(16) unsigned char adj_smem[];
  using Sh = AdjShared<T, FAM, D, G>;
  Sh& sh = *reinterpret_cast<Sh*>(adj_smem);
  constexpr int HV = hist_vals<FAM>();
  const int tid = threadIdx.x, lane = tid & 31, wg = tid >> 5;
  const int gl = tid, j = gl + 1;                 // this lane's node
  const int N = a.N;
  const bool mine = j <= N;
  const bool own0 = gl < D;                       // coordinate gl of node 0
  const int k0 = own0 ? gl : 0;
  const QCPar qp{a.qc_m, a.qc_ah, a.qc_gz, a.qc_eps};
  const T sig = a.sig, tau = a.tau, th = a.th;
  const size_t state = (size_t)3 * (N + 1) * D;   // one checkpoint
  T* work = a.work + (size_t)blockIdx.x * a.work_per_cta;
  // the segment's history after the checkpoints: per step a row of HV values per
  // lane, then D values of the new x_0 (each row a multiple of 16 bytes)
  T* hist = work + a.hist_off;
  const size_t hrow = (size_t)32 * G * HV + 16;
  const T ginv = T(1.0 / (1.0 + (double)tau * a.W2[k0]));
  const T goff = T((double)tau * a.W2[k0] * a.c[k0]) * ginv;
  if (own0) sh.c[k0] = a.c[k0];                   // each lane reads back its own

  for (;;) {
    __syncthreads();
    if (tid == 0) sh.item = atomicAdd(a.counter, 1ull);
    __syncthreads();
    const int64_t b = (int64_t)sh.item;
    if (b >= a.B) break;
    const int K = a.iters[b];
    if (K < 0 || K > a.K_cap) {
      if (tid == 0)
        for (int k = 0; k < D; ++k) a.dxq[b * D + k] = __longlong_as_double(0x7ff8000000000000ll);
      continue;
    }
    const double delta_d = a.t[b] / N;
    const T delta = T(a.t[b]) / T(N);
    const T L = sig * delta, taud = tau * delta;
    const uint64_t gid = (uint64_t)(a.point_offset + b);

    // ---- state of this lane: node j (x, p, z), and coordinate k0 of node 0
    T x[D], p[D], z[D], x0, z0;
    const InitGuess<T> ig(a.radius);                // the solver's initial guess
#pragma unroll
    for (int k = 0; k < D; ++k) {
      const double xq = a.xq[b * D + k];
      x[k] = (j < N) ? ig.x(xq, a.seed, gid, j, k) : T(xq);
      p[k] = mine ? ig.p(a.seed, gid, j, k) : T(0);
      z[k] = x[k];
    }
    x0 = ig.x(a.xq[b * D + k0], a.seed, gid, 0, k0);
    z0 = x0;

    // one forward iteration (the solver's step, one node per lane); hrow_k: where
    // the step leaves its history, or null
    auto step = [&](T* hrow_k) {
      slot_store<T, D>(sh.zs[gl], z);
      if (own0) sh.node0[k0] = z0;
      __syncthreads();
      T zl[D];
      slot_load<T, D>(gl > 0 ? sh.zs[gl - 1] : sh.node0, zl);
      T pn[D];
      QCNode<T> nd;
      if (mine) {
        T v[D];
        [[maybe_unused]] T hist_v[16];
        {
          T dz[D];
          v_sub<T, D>(dz, z, zl);
          v_fma<T, D>(v, sig, dz, p);                    // p + sigma (z_j - z_{j-1})
        }
        if constexpr (FAM == 1) {
          if (hrow_k != nullptr) {
            hist_v[0] = x[3]; hist_v[1] = x[4]; hist_v[2] = x[5];
            hist_v[3] = v[6]; hist_v[4] = v[7]; hist_v[5] = v[8];
          }
          qc_node<T>(reinterpret_cast<const T(&)[12]>(x), nd);
          qc_prox<T>(nd, qp, L, reinterpret_cast<const T(&)[12]>(x), reinterpret_cast<const T(&)[12]>(v),
                     reinterpret_cast<T(&)[12]>(pn));
          if (hrow_k != nullptr) {
#pragma unroll
            for (int k = 0; k < 6; ++k) hist_v[6 + k] = pn[k];
            hist_v[12] = pn[9]; hist_v[13] = pn[10]; hist_v[14] = pn[11]; hist_v[15] = T(0);
            constexpr int E = 16 / (int)sizeof(T);   // values per chunk
#pragma unroll
            for (int q = 0; q < hist_chunks<T, FAM>(); ++q) {
              T c[E];
#pragma unroll
              for (int e = 0; e < E; ++e) c[e] = hist_v[q * E + e];
              slot_store<T, E>(hrow_k + (size_t)(q * 32 * G + gl) * E, c);
            }
          }
        } else {
#pragma unroll
          for (int k = 0; k < D; ++k) pn[k] = v[k] / (T(1) + L);
        }
      } else {
#pragma unroll
        for (int k = 0; k < D; ++k) pn[k] = T(0);
      }
      slot_store<T, D>(sh.ps[gl], pn);
      __syncthreads();
      if (own0) {
        const T xn = (x0 + tau * sh.ps[0][k0]) * ginv + goff;
        z0 = xn + th * (xn - x0);
        x0 = xn;
        if (hrow_k != nullptr) hrow_k[(size_t)32 * G * HV + k0] = xn;
      }
      if (mine && j < N) {
        T g[D], pr[D];
        slot_load<T, D>(sh.ps[gl + 1], pr);
        if constexpr (FAM == 1) {
          qc_gradx<T>(nd, qp, reinterpret_cast<const T(&)[12]>(pn), reinterpret_cast<T(&)[12]>(g));
        } else {
#pragma unroll
          for (int k = 0; k < D; ++k) g[k] = T(0);
        }
        T dp[D], t[D], xn[D];
        v_sub<T, D>(dp, pn, pr);
        v_fma<T, D>(t, -tau, dp, x);
        v_fma<T, D>(xn, taud, g, t);                     // x - tau (p_j - p_{j+1}) + tau delta g
        v_sub<T, D>(t, xn, x);
        v_fma<T, D>(z, th, t, xn);
#pragma unroll
        for (int k = 0; k < D; ++k) x[k] = xn[k];
      }
#pragma unroll
      for (int k = 0; k < D; ++k) p[k] = pn[k];
    };
    auto save = [&](int slot) {
      T* s = work + (size_t)slot * state;
      if (mine)
#pragma unroll
        for (int k = 0; k < D; ++k) {
          s[(size_t)j * D + k] = x[k];
          s[(size_t)(N + 1) * D + (size_t)j * D + k] = p[k];
          s[(size_t)2 * (N + 1) * D + (size_t)j * D + k] = z[k];
        }
      if (own0) {
        s[k0] = x0;
        s[(size_t)2 * (N + 1) * D + k0] = z0;
      }
    };
    auto load = [&](int slot) {
      const T* s = work + (size_t)slot * state;
      if (mine)
#pragma unroll
        for (int k = 0; k < D; ++k) {
          x[k] = s[(size_t)j * D + k];
          p[k] = s[(size_t)(N + 1) * D + (size_t)j * D + k];
          z[k] = s[(size_t)2 * (N + 1) * D + (size_t)j * D + k];
        }
      if (own0) {
        x0 = s[k0];
        z0 = s[(size_t)2 * (N + 1) * D + k0];
      }
    };

    // ---- forward with checkpoints; the last piece (up to S steps) of the last segment
    // leaves its history at once.  kb: first iteration of the segment at hand, ks: of
    // the piece whose history is in the buffer.
    int kb = K > 0 ? (K - 1) / a.C * a.C : 0;
    int ks = K > 0 ? kb + (K - 1 - kb) / a.S * a.S : 0;
    for (int k = 0, next = 0, slot = 0, gap = a.C; k < K; ++k) {   // next: that of the next checkpoint
      if (k == kb) { next = kb; slot = a.slot_s; gap = a.S; }
      if (k == next && k < ks) { save(slot++); next += gap; }
      step(k >= ks ? hist + (size_t)(k - ks) * hrow : nullptr);
    }
    __syncthreads();

    // ---- adjoint of the value at s^K
    QCStep<T> steps;
    if (FAM == 1) sh.sums[gl] = QCSums{0.0, 0.0, 0.0, 0.0, 0.0};   // each lane's own
    double sW = 0.0, sc = 0.0;                       // coordinate k0 of node 0
    T xb[D], pb[D], zb[D], x0b = T(0), z0b = T(0);
    {
      slot_store<T, D>(sh.ps[gl], p);
      slot_store<T, D>(sh.zs[gl], x);
      if (own0) sh.node0[k0] = x0;
      __syncthreads();
      T gx[D], gp[D], pr[D], xl[D];
      QCNode<T> nd;
      double parb[4] = {0, 0, 0, 0};
      if (mine) {
        if constexpr (FAM == 1) {
          qc_node<T>(reinterpret_cast<const T(&)[12]>(x), nd);
          qc_gradx<T>(nd, qp, reinterpret_cast<const T(&)[12]>(p), reinterpret_cast<T(&)[12]>(gx));
          qc_gradp<T>(nd, qp, reinterpret_cast<const T(&)[12]>(x), reinterpret_cast<const T(&)[12]>(p),
                      reinterpret_cast<T(&)[12]>(gp));
          double hp[4];
          qc_dHdpar<T>(nd, qp, reinterpret_cast<const T(&)[12]>(p), hp);
          for (int i = 0; i < 4; ++i) parb[i] += -delta_d * hp[i];
        } else {
          for (int k = 0; k < D; ++k) { gx[k] = T(0); gp[k] = p[k]; }
        }
      }
      for (int i = 0; i < 4; ++i) {
        parb[i] = warp_sum<double>(parb[i]);
        if (lane == 0) sh.vpar[wg][i] = parb[i];
      }
      slot_load<T, D>(sh.ps[(mine && j < N) ? gl + 1 : gl], pr);
      slot_load<T, D>(gl > 0 ? sh.zs[gl - 1] : sh.node0, xl);
#pragma unroll
      for (int k = 0; k < D; ++k) {
        const T prk = (mine && j < N) ? pr[k] : T(0);
        xb[k] = mine ? (p[k] - prk - delta * gx[k]) : T(0);    // node N: p_N - delta grad_x H
        pb[k] = mine ? (x[k] - xl[k] - delta * gp[k]) : T(0);
        zb[k] = T(0);
      }
      if (own0) {
        const double e = (double)x0 - sh.c[k0];
        x0b = T(a.W2[k0] * e) - sh.ps[0][k0];                    // grad g(x_0) - p_1
        sh.W0[k0] = a.W[k0] * e * e;
        sh.c0[k0] = -a.W2[k0] * e;
      }
    }

    // ---- backward sweep, newest piece first; kend: the iterations not yet transposed
    for (int kend = K; kend > 0; kend = ks) {
      __syncthreads();                                // the slots are free again
      if (kend < K) {
        int k, next = kend, slot = a.slot_s;
        if (ks > kb) {                                // the piece before, of the same segment
          k = ks -= a.S;
          load(a.slot_s + (ks - kb) / a.S);
        } else {                                      // the last piece of the segment before
          k = next = kb -= a.C;
          ks = kb + (a.C - 1) / a.S * a.S;
          load(kb / a.C);
        }
        for (; k < kend; ++k) {
          if (k == next && k < ks) { save(slot++); next += a.S; }
          step(k >= ks ? hist + (size_t)(k - ks) * hrow : nullptr);
        }
        __syncthreads();
      }
      const int n = kend - ks;
      auto fetch = [&](int r, int buf) {              // history of the piece's step r
        if constexpr (FAM == 1) {
          if (mine) {
            const char* s = reinterpret_cast<const char*>(hist + (size_t)r * hrow) + 16 * gl;
            char* d = reinterpret_cast<char*>(sh.hist[buf][gl]);
#pragma unroll
            for (int q = 0; q < hist_chunks<T, FAM>(); ++q)
              cp_async16(d + 16 * q, s + (size_t)q * 32 * G * 16);
          }
        }
        cp_async_commit();
      };
      __threadfence();                                // the history is in memory before it is fetched
      fetch(n - 1, (n - 1) & 1);
      T x0p = own0 ? hist[(size_t)(n - 1) * hrow + (size_t)32 * G * HV + k0] : T(0);
      for (int r = n - 1; r >= 0; --r) {
        T x0p_next = T(0);
        if (r > 0) {
          fetch(r - 1, (r - 1) & 1);
          if (own0) x0p_next = hist[(size_t)(r - 1) * hrow + (size_t)32 * G * HV + k0];
          cp_async_wait<1>();
        } else {
          cp_async_wait<0>();
        }
        // intermediates of the step at s^k
        [[maybe_unused]] T v[D], pn[D];
        QCNode<T> nd;
        if constexpr (FAM == 1) {
          if (mine) {
            T h[16], xk[D], pl[D];
            slot_load<T, 16>(sh.hist[r & 1][gl], h);
#pragma unroll
            for (int kk = 0; kk < D; ++kk) { xk[kk] = T(0); v[kk] = T(0); }
            xk[3] = h[0]; xk[4] = h[1]; xk[5] = h[2];
            v[6] = h[3]; v[7] = h[4]; v[8] = h[5];
            qc_node<T>(reinterpret_cast<const T(&)[12]>(xk), nd);
            // rows 6-8 of p^{k+1} again; the other rows as the step left them
            qc_prox<T>(nd, qp, L, reinterpret_cast<const T(&)[12]>(xk),
                       reinterpret_cast<const T(&)[12]>(v), reinterpret_cast<T(&)[12]>(pl));
#pragma unroll
            for (int kk = 0; kk < D; ++kk)
              pn[kk] = kk < 6 ? h[6 + kk] : (kk < 9 ? pl[kk] : h[3 + kk]);
          }
        }
        // (xb, pb, zb) are the adjoints of s^{k+1}; build those of s^k
        T nxb[D], npb[D], nzb[D], pnb[D];
#pragma unroll
        for (int kk = 0; kk < D; ++kk) { nxb[kk] = T(0); npb[kk] = T(0); nzb[kk] = T(0); pnb[kk] = pb[kk]; }
        T xpb[D];                                     // adjoint of x^{k+1}_j after z' = x' + th (x' - x)
        if (mine && j < N) {
          v_fma<T, D>(xpb, T(1) + th, zb, xb);
          v_fma<T, D>(nxb, -th, zb, xpb);
          v_fma<T, D>(pnb, -tau, xpb, pb);
          T gb[D];
#pragma unroll
          for (int kk = 0; kk < D; ++kk) gb[kk] = taud * xpb[kk];
          if constexpr (FAM == 1)
            qc_gradx_vjp<T>(nd, qp, reinterpret_cast<const T(&)[12]>(pn), reinterpret_cast<const T(&)[12]>(gb),
                            reinterpret_cast<T(&)[12]>(nxb), reinterpret_cast<T(&)[12]>(pnb), steps,
                            sh.sums[gl]);
        } else {
#pragma unroll
          for (int kk = 0; kk < D; ++kk) xpb[kk] = T(0);
          if (mine)                                   // node N: x' = x, z' = x
#pragma unroll
            for (int kk = 0; kk < D; ++kk) nxb[kk] += xb[kk] + zb[kk];
        }
        // p'_{j} also enters x'_{j-1} (+tau) and, for j = 1, x'_0
        {
          T tx[D];
#pragma unroll
          for (int kk = 0; kk < D; ++kk) tx[kk] = tau * xpb[kk];
          slot_store<T, D>(sh.ps[gl], tx);
        }
        if (own0) {
          // x0' = (x0 + tau p'_1) ginv + goff; z0' = x0' + th (x0' - x0)
          const T x0pb = x0b + (T(1) + th) * z0b;
          const T nx0b = -th * z0b + x0pb * ginv;
          sh.node0[k0] = x0pb * ginv;
          sW += (double)x0pb * (sh.c[k0] - (double)x0p);
          sc += (double)x0pb;
          x0b = nx0b;
        }
        __syncthreads();
        if (mine && gl > 0) {
          T t[D];
          slot_load<T, D>(sh.ps[gl - 1], t);
#pragma unroll
          for (int kk = 0; kk < D; ++kk) pnb[kk] += t[kk];
        }
        if (gl == 0) {
          T t[D];
          slot_load<T, D>(sh.node0, t);
#pragma unroll
          for (int kk = 0; kk < D; ++kk) pnb[kk] += t[kk] * tau;
        }
        // dual step: p'_j = prox(x_j, v_j), v_j = p_j + sig (z_j - z_{j-1})
        T vb[D];
#pragma unroll
        for (int kk = 0; kk < D; ++kk) vb[kk] = T(0);
        if (mine) {
          if constexpr (FAM == 1)
            qc_prox_vjp<T>(nd, qp, L, reinterpret_cast<const T(&)[12]>(v), reinterpret_cast<const T(&)[12]>(pn),
                           reinterpret_cast<const T(&)[12]>(pnb), reinterpret_cast<T(&)[12]>(vb),
                           reinterpret_cast<T(&)[12]>(nxb), steps, sh.sums[gl]);
          else
#pragma unroll
            for (int kk = 0; kk < D; ++kk) vb[kk] = pnb[kk] / (T(1) + L);
#pragma unroll
          for (int kk = 0; kk < D; ++kk) { npb[kk] += vb[kk]; nzb[kk] += sig * vb[kk]; }
        }
        {
          T tv[D];
#pragma unroll
          for (int kk = 0; kk < D; ++kk) tv[kk] = -sig * vb[kk];
          slot_store<T, D>(sh.zs[gl], tv);
        }
        __syncthreads();
        if (mine && j < N) {
          T t[D];
          slot_load<T, D>(sh.zs[gl + 1], t);
#pragma unroll
          for (int kk = 0; kk < D; ++kk) nzb[kk] += t[kk];
        }
        if (own0) z0b = sh.zs[0][k0];
#pragma unroll
        for (int kk = 0; kk < D; ++kk) { xb[kk] = nxb[kk]; pb[kk] = npb[kk]; zb[kk] = nzb[kk]; }
        x0p = x0p_next;
        if constexpr (FAM == 1) {
          if (r % kHistSteps == 0) {                  // StepSum's bound is for 64 steps
            QCSums& q = sh.sums[gl];
            q.ma += steps.ma.take(); q.mc += steps.mc.take(); q.ah += steps.ah.take();
            q.gz += steps.gz.take(); q.eps += steps.eps.take();
          }
        }
      }
    }

    // ---- s^0 depends on x through x^0_j = x + r u (j < N), x^0_N = x, z^0 = x^0
    __syncthreads();
    if (own0) sh.node0[k0] = T(0);                    // (keeps the slot defined for the next point)
    const double wb = a.w[b];
    double parb[4] = {0, 0, 0, 0};
    if (FAM == 1) qc_par(sh.sums[gl], qp, parb);
    const double head = own0 ? (double)x0b + (double)z0b : 0.0;
#pragma unroll
    for (int k = 0; k < D; ++k) {
      double xqb = mine ? (double)xb[k] + (double)zb[k] : 0.0;
      if (gl == k) xqb += head;
      xqb = warp_sum<double>(xqb);
      if (lane == 0) sh.red[wg][k] = xqb;
    }
    for (int i = 0; i < 4; ++i) {
      parb[i] = warp_sum<double>(parb[i]);
      if (lane == 0) sh.red[wg][D + i] = parb[i];
    }
    __syncthreads();
    if (own0) {
      double s = 0.0;
      for (int w = 0; w < G; ++w) s += sh.red[w][k0];
      a.dxq[b * D + k0] = wb * s;
      const double Wb = sh.W0[k0] + sW * 2.0 * (double)tau * a.W[k0] * (double)ginv;
      const double cb = sh.c0[k0] + sc * (double)tau * a.W2[k0] * (double)ginv;
      atomicAdd(&a.dW[k0], wb * Wb);
      atomicAdd(&a.dc[k0], wb * cb);
    }
    if (FAM == 1 && gl >= 16 && gl < 20) {
      const int i = gl - 16;
      double s = 0.0;
      for (int w = 0; w < G; ++w) s += sh.red[w][D + i] + sh.vpar[w][i];
      atomicAdd(&a.ddyn[i], wb * s);
    }
  }
}

// Everything a launch of one instantiation needs: kernel, threads, shared memory,
// and the workspace of one CTA for (K_cap, C).
template <typename T, int FAM, int D, int G>
hj_status launch_adj_g(AdjArgs<T>& a, cudaStream_t s) {
  using Sh = AdjShared<T, FAM, D, G>;
  // FP64 quadcopter beyond 128 nodes: outside the entry point's range, not built
  if constexpr (sizeof(T) == 8 && D == 12 && G == 8) {
    return HJ_ERR_UNSUPPORTED;
  } else {
    auto kern = adjoint_kernel<T, FAM, D, G>;
    constexpr int smem = (int)sizeof(Sh);
    int dev = 0, nsm = 0, per_sm = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
        cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, 32 * G, smem) != cudaSuccess)
      return HJ_ERR_CUDA;
    // steps whose history is kept: the whole segment up to 64 (C is not above K_cap here),
    // beyond that 64, or about sqrt(C) where checkpoints every 64 steps would be the more
    a.S = a.C;
    if (a.C > kHistSteps) {
      a.S = kHistSteps;
      while ((int64_t)a.S * a.S < a.C) ++a.S;
    }
    a.slot_s = a.K_cap / a.C + 1;
    const int n_s = a.S < a.C ? (a.C - 1) / a.S + 1 : 0;
    const size_t ckpt = (((size_t)a.slot_s + n_s) * 3 * (a.N + 1) * D + 15) / 16 * 16;
    const size_t hrow = (size_t)32 * G * hist_vals<FAM>() + 16;
    a.hist_off = ckpt;
    a.work_per_cta = ckpt + (size_t)a.S * hrow;
    int64_t grid = (int64_t)nsm * (per_sm > 0 ? per_sm : 1);
    if (a.B < grid) grid = a.B;
    // fewer CTAs where the device has no room for all of them
    void* work = nullptr;
    while (cudaMalloc(&work, a.work_per_cta * sizeof(T) * (size_t)grid) != cudaSuccess) {
      (void)cudaGetLastError();
      work = nullptr;
      if (grid == 1) return HJ_ERR_OOM;
      grid = (grid + 1) / 2;
    }
    a.work = static_cast<T*>(work);
    hj_status r = HJ_OK;
    if (cudaMemsetAsync(a.counter, 0, sizeof(unsigned long long), s) != cudaSuccess) {
      r = HJ_ERR_CUDA;
    } else {
      kern<<<(int)grid, 32 * G, smem, s>>>(a);
      if (cudaGetLastError() != cudaSuccess) r = HJ_ERR_CUDA;
    }
    if (cudaStreamSynchronize(s) != cudaSuccess && r == HJ_OK) r = HJ_ERR_CUDA;
    cudaFree(work);
    return r;
  }
}

template <typename T, int FAM, int D>
hj_status launch_adj(AdjArgs<T>& a, cudaStream_t s) {
  switch ((a.N + 31) / 32) {
    case 1: return launch_adj_g<T, FAM, D, 1>(a, s);
    case 2: return launch_adj_g<T, FAM, D, 2>(a, s);
    case 3: case 4: return launch_adj_g<T, FAM, D, 4>(a, s);
    case 5: case 6: case 7: case 8: return launch_adj_g<T, FAM, D, 8>(a, s);
    default: return HJ_ERR_UNSUPPORTED;
  }
}

}  // namespace

template <typename T>
hj_status launch_adjoint(int family, const AdjArgs<T>& args, cudaStream_t s) {
  AdjArgs<T> a = args;
  if (a.C > a.K_cap) a.C = a.K_cap > 0 ? a.K_cap : 1;   // one segment either way
  if (a.N < 1 || a.N > 256) return HJ_ERR_UNSUPPORTED;
  if (family == HJ_FAMILY_QUADCOPTER && a.d == 12) return launch_adj<T, 1, 12>(a, s);
  if (family == HJ_FAMILY_QUADRATIC) {
    switch (a.d) {
      case 1: return launch_adj<T, 0, 1>(a, s);
      case 2: return launch_adj<T, 0, 2>(a, s);
      case 3: return launch_adj<T, 0, 3>(a, s);
      case 4: return launch_adj<T, 0, 4>(a, s);
      default: return HJ_ERR_UNSUPPORTED;
    }
  }
  return HJ_ERR_UNSUPPORTED;
}

template hj_status launch_adjoint<float>(int, const AdjArgs<float>&, cudaStream_t);
template hj_status launch_adjoint<double>(int, const AdjArgs<double>&, cudaStream_t);

}  // namespace hj
