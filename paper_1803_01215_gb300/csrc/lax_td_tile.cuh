// Register-tiled batched PDHG for the tanh-drift Hamiltonian with FP32 iterates:
// H = <p, tanh(A x)> + |p|^2/2 (Algorithm 1 with the Section 5.3 updates).
//
// A group of G warps (as many as the tiles need) solves one query point.  Each thread
// owns a fixed tile of 4 coordinates x TJ time nodes (TJ = 4 for d <= 64: 128 registers,
// twice the warps per SM, groups of up to 16 warps; TJ = 8 above, where the larger groups
// measured slower) and keeps that tile's x, p and z in registers
// for the whole solve (thread t of the group: j-tiles in blocks of 4, the last block
// as wide as it has tiles; within a block i-tile = u / width and j-tile = u % width, so a
// quarter-warp covers 2 i-tiles x 4 j-tiles).  Only
// what other threads need goes through shared memory:
//   Xs[k][j-1]   the x iterate of nodes 1..N (operand of A x), published after
//                the primal step;
//   Ws[k][j-1]   W = (1 - a^2) p (operand of A^T W), published after the dual step;
//   Zb, Pb       the z of each tile's last node and the p of its first node,
//                the neighbour terms z_{j-1} and p_{j+1} across tile boundaries.
// Per iteration:
//   phase A  Y = A X over the tile (k-loop over 16-byte loads of A^T and Xs),
//            then a = tanh(Y), the dual prox
//            p_j <- (p_j + sigma (z_j - z_{j-1}) - lam a) / (1 + lam), lam = sigma delta,
//            and W = (1 - a^2) p_j;
//   phase B  G = A^T W, then x_j <- x_j - tau (p_j - p_{j+1}) + tau delta G_j,
//            z_j = x_j + theta (x_j - x_j_old), and the g-prox of x_0 (held by
//            the threads of the first node tile).
// x_N stays pinned at the query point.  One group barrier after each phase
// (__syncwarp when G = 1).  On test iterations each thread's squared
// increments (its tile, FP32) are reduced over the warp in FP32, and the
// group's warp sums are accumulated as double-floats (error-free TwoSum: as
// accurate as FP64) and compared with tol; the value's (coordinate, node) terms
// are FP32 and their sum FP64.  Groups take points from the work
// counter (persistent grid); the CTA's groups share one copy of A and A^T.
//
// Row strides are compile-time (DP of A, NS of Xs and Ws, by classes of d and N), so the
// product's loads are immediate offsets.  Nothing in an iteration asks whether a row or a
// node exists: padding rows hold zeros and stay zero (no drift, no cost), and a column
// past N touches no other column; x_j keeps its value for j >= N by one select.
// Measured against the guards and run-time strides: d = 32, N = 32 (16384 points) 31.1 ->
// 25.8 ms, d = 100 (4096) 76.6 -> 65.6 ms; warps by the tiles instead of a power of two:
// d = 37, N = 24 (1500) 4.7 -> 2.9 ms.
#pragma once
#include <cuda_runtime.h>

#include "hj_internal.cuh"

namespace hj {

constexpr int kTI = 4;   // coordinates per tile

template <int DP, int NS>
struct TileLayout {
  int d, dp, TIc, TJc;
  size_t head_bytes;     // per-group item slots, g-prox and Hopf node-1 constants
  size_t a_floats;       // A^T and A
  size_t grp_floats;     // Xs, Ws, Zb, Pb, reductions of one group
  __host__ __device__ TileLayout(int d_, int Nmax, int TJ, int G, int M) {
    d = d_;
    dp = (d + 3) & ~3;
    TIc = dp / kTI;
    TJc = (Nmax + TJ - 1) / TJ;
    head_bytes = (size_t)((M * 8 + 15) / 16) * 16 + 4 * (size_t)dp * sizeof(float);
    a_floats = 2 * (size_t)d * DP;
    grp_floats = 2 * (size_t)dp * NS + 2 * (size_t)TJc * dp + 6 * (size_t)G;   // + 3G doubles
    grp_floats = (grp_floats + 3) & ~size_t(3);       // keep 16-byte alignment
  }
  __host__ __device__ size_t bytes(int M) const {
    return head_bytes + (a_floats + (size_t)M * grp_floats) * sizeof(float);
  }
};

// barrier of a group of G warps (G = 1: one warp)
__device__ __forceinline__ void group_barrier(int grp, int G) {
  if (G == 1) __syncwarp();
  else asm volatile("bar.sync %0, %1;" ::"r"(grp + 1), "r"(32 * G) : "memory");
}

template <int TJ>
__device__ __forceinline__ void storev(float* p, const float (&v)[TJ]) {
#pragma unroll
  for (int q = 0; q < TJ / 4; ++q)
    *reinterpret_cast<float4*>(p + 4 * q) = make_float4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
}

// acc[r][c] = sum_k M[k][i0 + r] * S[k][c0 + c], k < d (M k-major with stride DP, S with
// stride NS).  The accumulators are updated in pairs of nodes by the packed FP32 fma
// (__ffma2_rn: each lane rounded once, bitwise the same as two fmaf), half the
// issue slots of scalar fmaf.
template <int TJ, int DP, int NS>
__device__ __forceinline__ void tile_product(const float* M, const float* S, int d, int i0, int c0,
                                             float (&acc)[kTI][TJ]) {
  float2 acc2[kTI][TJ / 2];
#pragma unroll
  for (int r = 0; r < kTI; ++r)
#pragma unroll
    for (int q = 0; q < TJ / 2; ++q) acc2[r][q] = make_float2(0.f, 0.f);
  const float* mp = M + i0;
  const float* sp = S + c0;
  auto kstep = [&](int o) {
    const float4 a = *reinterpret_cast<const float4*>(mp + o * DP);
    float2 s2[TJ / 2];
#pragma unroll
    for (int q = 0; q < TJ / 4; ++q) {
      const float4 v = *reinterpret_cast<const float4*>(sp + o * NS + 4 * q);
      s2[2 * q] = make_float2(v.x, v.y);
      s2[2 * q + 1] = make_float2(v.z, v.w);
    }
    const float av[kTI] = {a.x, a.y, a.z, a.w};
#pragma unroll
    for (int r = 0; r < kTI; ++r) {
      const float2 ar = make_float2(av[r], av[r]);
#pragma unroll
      for (int q = 0; q < TJ / 2; ++q) acc2[r][q] = __ffma2_rn(ar, s2[q], acc2[r][q]);
    }
  };
  constexpr int U = 8;                     // k-steps per trip
  int k = 0;
#pragma unroll 1
  for (; k + U <= d; k += U) {
#pragma unroll
    for (int o = 0; o < U; ++o) kstep(o);
    mp += U * DP;
    sp += U * NS;
  }
  if (k + 4 <= d) {
#pragma unroll
    for (int o = 0; o < 4; ++o) kstep(o);
    mp += 4 * DP;
    sp += 4 * NS;
    k += 4;
  }
#pragma unroll 1
  for (; k < d; ++k) {
    kstep(0);
    mp += DP;
    sp += NS;
  }
#pragma unroll
  for (int r = 0; r < kTI; ++r)
#pragma unroll
    for (int q = 0; q < TJ / 2; ++q) { acc[r][2 * q] = acc2[r][q].x; acc[r][2 * q + 1] = acc2[r][q].y; }
}

// LAX1: the Lax form with theta = 1 (the paper's choice); else both are taken from the
// arguments.  Four-node tiles are held to 128 registers (CTAs of up to 512 threads,
// 16 warps per SM); eight-node tiles: up to 256 threads, about 240 registers.
template <int TJ, int DP, int NS, bool LAX1>
__global__ void __launch_bounds__(TJ == 4 ? 512 : 256, 1)
lax_td_tile_kernel(const SolveArgs<float> a, int G, int M) {
  constexpr int kTJ = TJ;
  extern __shared__ __align__(16) unsigned char smem[];
  const TileLayout<DP, NS> L(a.d, a.N, TJ, G, M);
  const int d = L.d, dp = L.dp;
  const bool HOPF = LAX1 ? false : a.formulation == HJ_FORM_HOPF;
  const bool TH1 = LAX1 ? true : a.theta == 1.0;
  unsigned long long* items = reinterpret_cast<unsigned long long*>(smem);
  float* goff = reinterpret_cast<float*>(smem + (size_t)((M * 8 + 15) / 16) * 16);
  float* ginv = goff + dp;
  float* hs = ginv + dp;                          // Hopf form: sigma / W^2 and sigma c
  float* hc = hs + dp;
  float* At = hc + dp;                            // At[k*DP + i] = A[i][k]
  float* Am = At + (size_t)d * DP;                // Am[k*DP + i] = A[k][i]
  const int grp = (int)threadIdx.x / (32 * G);
  float* Xs = Am + (size_t)d * DP + (size_t)grp * L.grp_floats;
  float* Ws = Xs + (size_t)dp * NS;
  float* Zb = Ws + (size_t)dp * NS;               // Zb[jt*dp + i]
  float* Pb = Zb + (size_t)L.TJc * dp;            // Pb[jt*dp + i]
  // [2G] floats (test sums, in the space of 2G doubles) then [G] doubles (value);
  // Pb + TJc dp floats keeps 16-byte alignment
  float* tred = Pb + (size_t)L.TJc * dp;
  double* vred = reinterpret_cast<double*>(tred) + 2 * G;

  for (int e = threadIdx.x; e < d * DP; e += blockDim.x) {
    const int k = e / DP, i = e - k * DP;
    At[e] = (i < d) ? a.At[k * d + i] : 0.f;
    Am[e] = (i < d) ? a.A[k * d + i] : 0.f;
  }
  for (int i = threadIdx.x; i < dp; i += blockDim.x) {
    const double w2 = i < d ? a.W2[i] : 0.0, cc = i < d ? a.c[i] : 0.0;
    goff[i] = (float)(a.tau * w2 * cc);
    ginv[i] = (float)(1.0 / (1.0 + a.tau * w2));
    hs[i] = (HOPF && i < d) ? (float)(a.sigma / w2) : 0.f;
    hc[i] = (float)(a.sigma * cc);
  }
  __syncthreads();

  const int t = (int)threadIdx.x - grp * 32 * G;  // thread within the group
  const int lane = t & 31, wig = t >> 5;
  const int blk = 4 * L.TIc;
  const int jg = t / blk, u = t - jg * blk;
  const int width = L.TJc - 4 * jg < 4 ? L.TJc - 4 * jg : 4;   // j-tiles of the block
  const bool tile_ok = width > 0 && u < width * L.TIc;
  const int it = tile_ok ? u / width : 0, jt = tile_ok ? 4 * jg + u % width : 0;
  const int i0 = it * kTI, c0 = jt * kTJ, j0 = 1 + c0;   // nodes j0..j0+TJ-1 <-> Xs columns c0..c0+TJ-1
  const float sig = a.sigma_t, tau = a.tau_t, th = a.theta_t;
  float4* zb_out = reinterpret_cast<float4*>(Zb + jt * dp + i0);
  float4* pb_out = reinterpret_cast<float4*>(Pb + jt * dp + i0);
  const float4* zb_in = reinterpret_cast<const float4*>(Zb + (jt > 0 ? jt - 1 : 0) * dp + i0);
  const float4* pb_in = reinterpret_cast<const float4*>(Pb + (jt + 1 < L.TJc ? jt + 1 : jt) * dp + i0);

  for (;;) {
    group_barrier(grp, G);
    if (t == 0) items[grp] = draw_item(a);
    group_barrier(grp, G);
    const int64_t item = (int64_t)items[grp];
    if (item >= a.B) break;
    const PointRef<float> ref = point_ref(a, item);
    const int64_t b = ref.id;
    const int N = ref.N;
    if (N < 1 || N > a.N) {                      // the host never routes such a point here
      if (t == 0) { a.status[b] = HJ_POINT_INVALID; a.iters[b] = 0; a.V[b] = 0.0; }
      continue;
    }
    const bool act = tile_ok && c0 < N;           // the tile holds nodes of this point
    const int nup = N - j0;                       // columns c < nup have j < N: their x moves
    const float delta_t = (float)a.t[b] / (float)N;
    const float lam = sig * delta_t, taud = tau * delta_t;
    const float ilam = 1.f / (1.f + lam);
    const uint64_t pt = (uint64_t)(a.point_offset + b);

    float x[kTI][kTJ], p[kTI][kTJ], z[kTI][kTJ], x0[kTI], z0[kTI];
    {
      const InitGuess<float> ig(a.radius);
#pragma unroll
      for (int r = 0; r < kTI; ++r) {
        const int i = i0 + r;
        const bool row = act && i < d;
        const double xq = row ? ref.xq[i] : 0.0;
#pragma unroll
        for (int c = 0; c < kTJ; ++c) {
          const int j = j0 + c;
          float xv = 0.f, pv = 0.f;
          if (row && j <= N) {
            if (a.warm_x == nullptr) {
              xv = (j < N) ? ig.x(xq, a.seed, pt, j, i) : (float)xq;
              pv = ig.p(a.seed, pt, j, i);
            } else {
              xv = (j < N) ? a.warm_x[ref.traj + (size_t)j * d + i] : (float)xq;
              pv = a.warm_p[ref.traj + (size_t)j * d + i];
            }
          }
          x[r][c] = xv; p[r][c] = pv; z[r][c] = xv;
        }
        float x0v = 0.f;                          // Hopf: x_0 is not a variable (0)
        if (row && jt == 0 && !HOPF)
          x0v = (a.warm_x == nullptr) ? ig.x(xq, a.seed, pt, 0, i) : a.warm_x[ref.traj + i];
        x0[r] = x0v; z0[r] = x0v;
      }
    }
    if (act) {
#pragma unroll
      for (int r = 0; r < kTI; ++r) storev<kTJ>(Xs + (size_t)(i0 + r) * NS + c0, x[r]);
      *zb_out = make_float4(z[0][kTJ - 1], z[1][kTJ - 1], z[2][kTJ - 1], z[3][kTJ - 1]);
    }
    group_barrier(grp, G);

    // one iteration; CHK adds the squared increments (test iterations only)
    auto step = [&](auto chk_tag, float& rx, float& rp) {
      constexpr bool CHK = decltype(chk_tag)::value;
      float acc[kTI][kTJ];
      // ---- phase A: Y = A X, tanh, dual prox, W = (1 - a^2) p
      if (act) {
        const float4 zq = *zb_in;
        const float zL[kTI] = {jt == 0 ? z0[0] : zq.x, jt == 0 ? z0[1] : zq.y,
                               jt == 0 ? z0[2] : zq.z, jt == 0 ? z0[3] : zq.w};
        tile_product<kTJ, DP, NS>(At, Xs, d, i0, c0, acc);
#pragma unroll
        for (int r = 0; r < kTI; ++r) {
          float w[kTJ];
#pragma unroll
          for (int c = 0; c < kTJ; ++c) {
            const float av = tanhf(acc[r][c]);
            const float zl = (c == 0) ? zL[r] : z[r][c - 1];
            const float v = p[r][c] + sig * (z[r][c] - zl);
            // fused by name: with lam a in both forms below the compiler rounds the product
            // first, and the two instantiations would not give the same bits
            float pn = fmaf(-lam, av, v) * ilam;
            if (!LAX1 && HOPF && c == 0 && jt == 0)  // Hopf node 1: prox of sigma g* + lam H
              pn = __fdividef(fmaf(-lam, av, v - hc[i0 + r]), 1.f + lam + hs[i0 + r]);
            if constexpr (CHK) { const float e = pn - p[r][c]; rp += (c <= nup) ? e * e : 0.f; }
            p[r][c] = pn;
            w[c] = (1.f - av * av) * pn;
          }
          storev<kTJ>(Ws + (size_t)(i0 + r) * NS + c0, w);
        }
        *pb_out = make_float4(p[0][0], p[1][0], p[2][0], p[3][0]);
      }
      group_barrier(grp, G);
      // ---- phase B: G = A^T W, primal gradient step, relaxation; g-prox of x_0
      if (act) {
        const float4 pq = *pb_in;                 // p_{j+1} of the tile's last column
        const float pR[kTI] = {pq.x, pq.y, pq.z, pq.w};
        tile_product<kTJ, DP, NS>(Am, Ws, d, i0, c0, acc);
#pragma unroll
        for (int r = 0; r < kTI; ++r) {
#pragma unroll
          for (int c = 0; c < kTJ; ++c) {
            const float pn = (c + 1 < kTJ) ? p[r][c + 1 < kTJ ? c + 1 : c] : pR[r];
            const float xo = x[r][c];
            const float xm = xo - tau * (p[r][c] - pn) + taud * acc[r][c];
            const float xn = (c < nup) ? xm : xo;
            if constexpr (CHK) { const float e = xn - xo; rx += e * e; }
            z[r][c] = TH1 ? 2.f * xn - xo : xn + th * (xn - xo);
            x[r][c] = xn;
          }
          if (jt == 0 && !HOPF) {                 // x_0 <- prox_{tau g}(x_0 + tau p_1)
            const float xo = x0[r];
            const float xn = (xo + tau * p[r][0] + goff[i0 + r]) * ginv[i0 + r];
            if constexpr (CHK) { const float e = xn - xo; rx += e * e; }
            z0[r] = TH1 ? 2.f * xn - xo : xn + th * (xn - xo);
            x0[r] = xn;
          }
          storev<kTJ>(Xs + (size_t)(i0 + r) * NS + c0, x[r]);
        }
        *zb_out = make_float4(z[0][kTJ - 1], z[1][kTJ - 1], z[2][kTJ - 1], z[3][kTJ - 1]);
      }
      group_barrier(grp, G);
    };

    int k_it = 0;
    int8_t st = HJ_POINT_MAX_ITER;
    const int max_iter = a.max_iter, check_every = a.check_every;
    while (k_it < max_iter) {
      const int left = max_iter - k_it;
      const int plain = (check_every - 1 < left - 1) ? check_every - 1 : left - 1;
      float dx = 0.f, dpp = 0.f;
      for (int r = 0; r < plain; ++r) step(std::integral_constant<bool, false>{}, dx, dpp);
      float rx = 0.f, rp = 0.f;
      step(std::integral_constant<bool, true>{}, rx, rp);
      k_it += plain + 1;
      // the threads' FP32 partials reduced over each warp in FP32; the group's
      // warp sums accumulated as double-floats (as accurate as FP64, on the
      // FP32 pipe) and compared with tol
      const float wx = warp_sum<float>(rx), wp = warp_sum<float>(rp);
      int verdict;                                // 1 converged, 2 non-finite
      if (G > 1) {
        if (lane == 0) { tred[2 * wig] = wx; tred[2 * wig + 1] = wp; }
        group_barrier(grp, G);
        verdict = stop_verdict<float>(a, tred, G, lane);
        group_barrier(grp, G);                    // tred is free for the next test
      } else {
        verdict = stop_verdict1<float>(a, wx, wp);
      }
      if (verdict == 2) { st = HJ_POINT_NONFINITE; break; }
      if (verdict == 1) { st = HJ_POINT_CONVERGED; break; }
    }

    // ---- value: g(x_0) + sum_j <p_j, x_j - x_{j-1}> - delta sum_j H(x_j, p_j); FP32
    // terms (A x from the FP32 copy of A), FP64 sum.  Xs holds the final x.
    double vacc = 0.0;
    if (act) {
      float acc[kTI][kTJ];
      tile_product<kTJ, DP, NS>(At, Xs, d, i0, c0, acc);
#pragma unroll
      for (int r = 0; r < kTI; ++r) {
        const int i = i0 + r;
        if (i < d) {
          const float xl0 = (jt == 0) ? x0[r] : Xs[(size_t)i * NS + c0 - 1];
#pragma unroll
          for (int c = 0; c < kTJ; ++c) {
            if (j0 + c <= N) {
              const float pv = p[r][c];
              const float dxv = x[r][c] - ((c == 0) ? xl0 : x[r][c > 0 ? c - 1 : 0]);
              vacc += (double)(pv * dxv - delta_t * (pv * tanhf(acc[r][c]) + 0.5f * pv * pv));
            }
          }
          if (jt == 0) {
            if (HOPF) {                           // -g*(p_1)
              const double p1 = (double)p[r][0];
              vacc -= p1 * a.c[i] + 0.5 * p1 * p1 / a.W2[i];
            } else {
              const double e = (double)x0[r] - a.c[i];
              vacc += 0.5 * a.W2[i] * e * e;
            }
          }
        }
      }
    }
    vacc = warp_sum<double>(vacc);
    if (G > 1) {
      if (lane == 0) vred[wig] = vacc;
      group_barrier(grp, G);
      vacc = 0.0;
      for (int w = 0; w < G; ++w) vacc += vred[w];
    }
    if (t == 0) {
      a.V[b] = vacc;
      a.iters[b] = k_it;
      a.status[b] = st;
      count_iterations(a, k_it);
    }
    if (act) {
#pragma unroll
      for (int r = 0; r < kTI; ++r) {
        const int i = i0 + r;
        if (i >= d) continue;
#pragma unroll
        for (int c = 0; c < kTJ; ++c) {
          const int j = j0 + c;
          if (j <= N) {
            if (a.traj_x != nullptr) a.traj_x[ref.traj + (size_t)j * d + i] = x[r][c];
            if (a.traj_p != nullptr) a.traj_p[ref.traj + (size_t)j * d + i] = p[r][c];
          }
        }
        if (jt == 0) {
          if (a.traj_x != nullptr)                // Hopf: x_0 = grad g*(p_1) = c + p_1 / W^2
            a.traj_x[ref.traj + i] = HOPF ? (float)(a.c[i] + (double)p[r][0] / a.W2[i]) : x0[r];
          if (a.traj_p != nullptr) a.traj_p[ref.traj + i] = 0.f;
        }
      }
    }
  }
}

template <int TJ, int DP, int NS, bool LAX1>
hj_status launch_tile_kernel(const SolveArgs<float>& a, cudaStream_t s) {
  auto kern = lax_td_tile_kernel<TJ, DP, NS, LAX1>;
  int dev = 0, nsm = 0, max_optin = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&max_optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess)
    return HJ_ERR_CUDA;
  // as many warps as the tiles fill, and one to four groups per CTA
  const int tiles = ((a.d + 3) / 4) * ((a.N + TJ - 1) / TJ);
  const int G = (tiles + 31) / 32;
  if (32 * G > (TJ == 4 ? 512 : 256)) return HJ_ERR_UNSUPPORTED;
  auto bytes = [&](int m) { return TileLayout<DP, NS>(a.d, a.N, TJ, G, m).bytes(m); };
  int M = G == 1 ? 4 : G == 2 ? 2 : 1;
  if (TJ == 8 && G <= 4) M = 8 / G;               // eight warps share one copy of A
  while (M > 1 && bytes(M) > (size_t)max_optin) M /= 2;
  // no second point on an SM while another SM has none (d = 100, N = 32: 152 points take
  // 6.27 ms two to a CTA, 3.92 one to a CTA; from 153 points on two, 200 points 7.06 ms)
  while (M > 1 && (int64_t)(M / 2) * nsm >= a.B) M /= 2;
  const size_t smem = bytes(M);
  if (smem > (size_t)max_optin) return HJ_ERR_UNSUPPORTED;
  if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess)
    return HJ_ERR_CUDA;
  const int threads = 32 * G * M;
  int bps = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&bps, kern, threads, smem) != cudaSuccess)
    return HJ_ERR_CUDA;
  if (bps < 1) return HJ_ERR_UNSUPPORTED;
  const int64_t ctas_needed = (a.B + M - 1) / M;
  const int64_t cap = (int64_t)bps * nsm;
  const int grid = (int)(ctas_needed < cap ? ctas_needed : cap);
  kern<<<grid, threads, smem, s>>>(a, G, M);
  return cudaGetLastError() == cudaSuccess ? HJ_OK : HJ_ERR_CUDA;
}

template <int TJ, int DP, int NS>
hj_status launch_tile(const SolveArgs<float>& a, cudaStream_t s) {
  return (a.theta == 1.0 && a.formulation != HJ_FORM_HOPF) ? launch_tile_kernel<TJ, DP, NS, true>(a, s)
                                                           : launch_tile_kernel<TJ, DP, NS, false>(a, s);
}

// d in a class of A's row stride; the row stride of Xs and Ws by N (lax_td_tile_*.cu)
hj_status launch_tile_d32(const SolveArgs<float>& a, cudaStream_t s);
hj_status launch_tile_d64(const SolveArgs<float>& a, cudaStream_t s);
hj_status launch_tile_d104(const SolveArgs<float>& a, cudaStream_t s);
hj_status launch_tile_d128(const SolveArgs<float>& a, cudaStream_t s);

}  // namespace hj
