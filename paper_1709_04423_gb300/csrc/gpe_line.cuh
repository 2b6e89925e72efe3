// gpe_line.cuh -- every time step of a 1d grid in one launch.
//
// A 1d line (Cartesian, the radial problem of a spherical trap, or the rho
// axis of a circular trap) is at most a few thousand points: one launch per
// step left it bound by the launch and by the serial recurrence of one warp
// (256-point lines) or of one thread (lines over 514 points).  Here the line
// stays in registers for the whole run: thread i of the launch owns S
// consecutive interior points, a block's warps and the blocks of one cluster
// follow each other along the line, and a step needs two exchanges (three in
// imaginary time) through shared memory -- one block's own, or, with more
// than one block, every block's, written through the cluster's distributed
// shared memory before its hardware barrier (no spin waits).
//
// The solve is the increment-form segment scan of gpe_sweep2.cuh with the
// thread's S points as the segment:
//   e_k = alpha_k (e_{k-1} + 2 p_k - p_{k-1} - p_{k+1}),  z_k = e_k + alpha_k z_{k+1},
//   u_k = p_k - 2 z_k     (half scale; a rho axis: its own coefficients),
// thread carries by a shuffle scan whose products do not change from step to
// step and are formed once per launch, warp carries from the published values
// of the warps before (after).  The first exchange carries a warp's first and
// last point and its forward end value formed without the two neighbouring
// points; their part enters linearly afterwards: with X = E - p_last of the
// warp before, every point adds G_k X (G_k the product of alpha from the
// warp's start to k) and the warp's last point takes -alpha p_first of the
// warp after.  Scans and carries are cut to the reach of the coefficients
// (`levels`, `depth`: products below 2^-48 for an FP32 state, 2^-64 otherwise),
// as in every other sweep.
//
// Points past the end of the line are zeros with zero coefficients, so the
// step loop has no bounds tests.  The double-float N reads its tables in the loop:
// a point past the end takes the last interior point's factor, not the end
// point's, where a potential may be infinite (a test there instead of the clamp:
// 513 points, imaginary time, 3.65 us per step against 3.61).
//
// Bound by latency: the chain of shuffles, barriers and (FP64) dependent FP64
// operations of one step; no memory traffic inside the loop.  Measured per
// step, against one launch per step before: 513 radial points FP32 10.5 -> 1.6
// us, 256 points FP64 17.6 -> 3.9 us (imaginary time); 4001 points FP64 real
// time 9.0 ms (one thread walked the line) -> 7.0 us.
#pragma once
#include "gpe_step.cuh"

namespace gpe {

constexpr int kLineMaxCtas = 16;                   // blocks of the cluster
constexpr int kLineMaxThreads = 512;
constexpr int kLineMaxWarps = kLineMaxCtas * kLineMaxThreads / 32;

template <typename T>
struct LineArgs {
  Sweep2Args<T> a;   // the state, coefficients, norm weights and the sub-step N of a step
  Sweep2Args<T> h;   // N(dt/2) of a real-time Strang run's first opening and last closing half
  long nsteps;
  int levels, depth;  // shuffle levels of the thread scan, warps a carry crosses
  int half_first;     // the first step opens with h (else a)
  int close_each;     // every step closes with a's N (imaginary-time Strang)
  int close_end;      // the run closes with h's N
};

__device__ __forceinline__ unsigned cluster_rank() {
  unsigned r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}

// Writes v at the address of block `rank` that corresponds to dst in this block's shared memory.
template <typename V>
__device__ __forceinline__ void st_cluster(V* dst, unsigned rank, V v) {
  static_assert(sizeof(V) == 4 || sizeof(V) == 8 || sizeof(V) == 16, "4, 8 or 16 bytes");
  static_assert(alignof(V) == sizeof(V), "one aligned vector store");
  unsigned a;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"((unsigned)__cvta_generic_to_shared(dst)), "r"(rank));
  unsigned w[sizeof(V) / 4];
  memcpy(w, &v, sizeof(V));
  if constexpr (sizeof(V) == 4) asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(a), "r"(w[0]) : "memory");
  else if constexpr (sizeof(V) == 8)
    asm volatile("st.shared::cluster.v2.u32 [%0], {%1, %2};" ::"r"(a), "r"(w[0]), "r"(w[1]) : "memory");
  else
    asm volatile("st.shared::cluster.v4.u32 [%0], {%1, %2, %3, %4};" ::"r"(a), "r"(w[0]), "r"(w[1]), "r"(w[2]),
                 "r"(w[3])
                 : "memory");
}

// 1/sqrt(s) = y0 (1 - r)^(-1/2) with the FP32 estimate y0 and r = 1 - s y0^2,
// about 2^-22: the binomial series to second order, y0 (1 + r/2 + 3 r^2/8) (the
// omitted term is below 2^-66); outside the FP32 range the library functions.
__device__ __forceinline__ double line_rsqrt(double s) {
  if (!(s > 1e-30 && s < 1e30)) return 1.0 / ::sqrt(s);
  const double y0 = (double)rsqrtf((float)s);
  const double r = ::fma(-s * y0, y0, 1.0);
  return ::fma(y0 * r, ::fma(0.375, r, 0.5), y0);
}
__device__ __forceinline__ df64 line_rsqrt(df64 s) {
  if (!(s.hi > 1e-30f && s.hi < 1e30f)) return df64(1.0 / ::sqrt((double)s));
  const float y0 = rsqrtf(s.hi);
  const df64 r = df64(1) - dfl::df_mulf(dfl::df_mulf(s, y0), y0);
  return df64(y0, 0.f) + dfl::df_mulf(dfl::df_scale(r, 0.5f) + df64(0.375f * r.hi * r.hi, 0.f), y0);
}

// The type a line's norm is summed in: the state precision (as a block's sums
// are in the other kernels), and SquareSum for FP32 lines of more than 514 points,
// the ones with several points per thread (as on the long lines of 2d and 3d
// grids; see flex_body).
template <typename T, int S>
using line_norm_t = typename std::conditional<std::is_same<T, float>::value && (S > 1), SquareSum, T>::type;

// The pending factor 1/sqrt(wscale * total) from the warps' norm sums in
// shared memory, by every warp for itself: in FP64 from FP64 sums, in
// double-float from the others (48 bits, on the FP32 pipes: a warp's FP64 chain
// would take longer than the rest of the step).
template <typename T>
using line_scale_t = typename std::conditional<std::is_same<T, double>::value, double, df64>::type;

__device__ __forceinline__ float line_factor(const SquareSum* nrm, int nparts, df64 ws) {
  const SquareSum t = SquareSum::gather(nrm, nparts);
  float h, l;
  dfl::df_two_sum(t.s, t.c, h, l);
  return line_rsqrt(df64(h, l + t.d) * ws).hi * SquareSum::pow2(-t.e);
}

template <typename T>
__device__ __forceinline__ T line_factor(const T* nrm, int nparts, line_scale_t<T> ws) {
  const int lane = threadIdx.x & 31;
  T s = T(0);
  for (int i = lane; i < nparts; i += 32) s = s + nrm[i];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1)
    if (o < nparts) s = s + shfl_xor_t(s, o);
  // (with fewer parts than lanes only the low lanes hold sums)
  if constexpr (std::is_same<T, double>::value) {
    return line_rsqrt(__shfl_sync(0xffffffffu, s, 0) * ws);
  } else if constexpr (std::is_same<T, float>::value) {
    return line_rsqrt(dfl::df_mulf(ws, __shfl_sync(0xffffffffu, s, 0))).hi;
  } else {
    const df64 t = df64(__shfl_sync(0xffffffffu, s.hi, 0), __shfl_sync(0xffffffffu, s.lo, 0));
    return line_rsqrt(t * ws);
  }
}

template <typename T, bool IMAG, bool VAR, int S>
__global__ void __launch_bounds__(kLineMaxThreads) line_steps_kernel(const __grid_constant__ LineArgs<T> P) {
  using c2 = c2_t<T>;
  __shared__ c2 s_first[kLineMaxWarps], s_last[kLineMaxWarps], s_end[kLineMaxWarps], s_z[kLineMaxWarps + 1];
  __shared__ c2 s_A[kLineMaxWarps], s_B[kLineMaxWarps], s_cr[kLineMaxWarps];
  using NT = line_norm_t<T, S>;
  __shared__ NT s_nrm[kLineMaxWarps];
  const Sweep2Args<T>& A = P.a;
  const int n = A.geom.n, M = n - 2;
  const int lane = threadIdx.x & 31, nw = blockDim.x >> 5;
  const int C = gridDim.x;
  const int rank = C > 1 ? (int)cluster_rank() : 0;
  const int w = rank * nw + (threadIdx.x >> 5), W = C * nw;  // this warp, warps along the line
  const int k0 = 1 + (w * 32 + lane) * S;
  const c2 zero = mk<T>(0, 0);
  // all blocks' shared memory written before the barrier is seen after it
  auto sync = [&]() {
    if (C > 1) {
      asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
    } else {
      __syncthreads();
    }
  };
  // lane src's value into entry i of every block's array
  auto publish = [&](auto* arr, int i, auto v) {
    if (C == 1) arr[i] = v;
    else if (lane < C) st_cluster(arr + i, (unsigned)lane, v);
  };
  auto bcast = [&](c2 v, int src) -> c2 {
    if constexpr (is_df<T>::value)
      return c2{df64(__shfl_sync(0xffffffffu, v.x.hi, src), __shfl_sync(0xffffffffu, v.x.lo, src)),
                df64(__shfl_sync(0xffffffffu, v.y.hi, src), __shfl_sync(0xffffffffu, v.y.lo, src))};
    else return mk<T>(__shfl_sync(0xffffffffu, v.x, src), __shfl_sync(0xffffffffu, v.y, src));
  };
  constexpr bool kF64 = std::is_same<T, double>::value;

  // ---- constants of this thread's points: coefficients, N, norm weights, the state
  c2 p[S], al[S], ab[VAR ? S : 1], bf[VAR ? S : 1], hh[VAR ? S : 1];
  T vk[is_df<T>::value ? 1 : S], gk[S], wk[IMAG ? S : 1];
#pragma unroll
  for (int j = 0; j < S; ++j) {
    const int k = k0 + j;
    const bool ok = k <= M;
    const int kc = ok ? k : 0;
    al[j] = ok ? A.alpha[kc] : zero;
    if constexpr (VAR) {
      ab[j] = ok ? A.vab[kc] : zero;
      bf[j] = ok ? A.vbf[kc] : zero;
      hh[j] = ok ? A.vh[kc] : zero;
    }
    p[j] = ok ? A.psi[kc] : zero;
    gk[j] = std::is_same<T, float>::value ? A.g : A.dtg;
    if (A.gw) gk[j] = gk[j] * A.gw[kc];
    if constexpr (!is_df<T>::value) vk[j] = !ok ? T(0) : A.V ? A.V[kc] : A.vx[kc] + (A.vy[0] + A.vz[0]);
    if constexpr (IMAG) wk[j] = ok ? A.w_axis[kc] : T(0);
  }
  // N of a step (dt, or dt/2 in imaginary-time Strang steps)
  auto phase = [&](c2 v, int j) -> c2 {
    const int k = min(k0 + j, M);
    if constexpr (is_df<T>::value) return phase_df<IMAG>(v, A, k, k, 0, gk[j]);
    else if constexpr (kF64) return phase_theta<IMAG>(v, fma(gk[j], fma(v.x, v.x, v.y * v.y), A.dt * vk[j]));
    else return phase_direct<T, IMAG>(v, vk[j], A.dt, gk[j]);
  };
  // N(dt/2) of a real-time Strang run's two ends
  auto phase_half = [&](c2 v, int j) -> c2 {
    const Sweep2Args<T>& H = P.h;
    const int k = min(k0 + j, M);
    if constexpr (is_df<T>::value) {
      return phase_df<IMAG>(v, H, k, k, 0, H.gw ? H.dtg * H.gw[k] : H.dtg);
    } else if constexpr (kF64) {  // (g dt/2 is exactly half of g dt)
      return phase_theta<IMAG>(v, fma(0.5 * gk[j], fma(v.x, v.x, v.y * v.y), H.dt * vk[j]));
    } else {
      return phase_direct<T, IMAG>(v, vk[j], H.dt, gk[j]);
    }
  };
  auto back = [&](int j) -> c2 { return VAR ? ab[VAR ? j : 0] : al[j]; };

  // products of the coefficients: within the thread (gf, gb), over the scan
  // levels (Pm, Qm), from the warp's start (end) to each point (gw, gbw)
  c2 gf[S], gb[S], gw[S], gbw[S], Pm[5], Qm[5];
  {
    c2 acc = al[0];
    gf[0] = acc;
#pragma unroll
    for (int j = 1; j < S; ++j) gf[j] = acc = cf_cc<T, IMAG>(acc, al[j]);
    acc = back(S - 1);
    gb[S - 1] = acc;
#pragma unroll
    for (int j = S - 2; j >= 0; --j) gb[j] = acc = cf_cc<T, IMAG>(acc, back(j));
    c2 a = gf[S - 1], b = gb[0], ia = a, ib = b;
#pragma unroll
    for (int l = 0; l < 5; ++l) {
      const int o = 1 << l;
      const c2 ua = shfl_up2<T>(a, o), ub = shfl_down2<T>(b, o), va = shfl_up2<T>(ia, o), vb = shfl_down2<T>(ib, o);
      Pm[l] = lane >= o ? a : zero;
      Qm[l] = lane + o < 32 ? b : zero;
      a = lane >= o ? cf_cc<T, IMAG>(a, ua) : zero;
      b = lane + o < 32 ? cf_cc<T, IMAG>(b, ub) : zero;
      if (lane >= o) ia = cf_cc<T, IMAG>(ia, va);
      if (lane + o < 32) ib = cf_cc<T, IMAG>(ib, vb);
    }
    c2 xa = shfl_up2<T>(ia, 1), xb = shfl_down2<T>(ib, 1);
    if (lane == 0) xa = mk<T>(1, 0);
    if (lane == 31) xb = mk<T>(1, 0);
#pragma unroll
    for (int j = 0; j < S; ++j) {
      gw[j] = cf_cc<T, IMAG>(gf[j], xa);
      gbw[j] = cf_cc<T, IMAG>(gb[j], xb);
    }
  }
  // the coefficient of the point after a thread's last one
  const c2 cr = VAR ? mk<T>(bf[VAR ? S - 1 : 0].x * hh[VAR ? S - 1 : 0].y, bf[VAR ? S - 1 : 0].y * hh[VAR ? S - 1 : 0].y)
                    : al[S - 1];
  if (C > 1) sync();  // every block of the cluster has started before its memory is written
  {
    const c2 wa = bcast(gw[S - 1], 31), wb = bcast(gbw[0], 0), wc = bcast(cr, 31);
    if (C > 1 || lane == 0) {
      publish(s_A, w, wa);
      publish(s_B, w, wb);
      publish(s_cr, w, wc);
    }
    if (threadIdx.x == 0) s_z[W] = zero;  // in this block's copy: nothing comes after the last warp
  }

  const line_scale_t<NT> ws(A.parts_wscale);
  for (long t = 0; t < P.nsteps; ++t) {
    // ---- the pending renormalisation and N
    if (IMAG && t > 0) {
      const T scl = line_factor(s_nrm, W, ws);
#pragma unroll
      for (int j = 0; j < S; ++j) {
        p[j].x = p[j].x * scl;
        p[j].y = p[j].y * scl;
      }
    }
    if (!IMAG && t == 0 && P.half_first) {
#pragma unroll
      for (int j = 0; j < S; ++j) p[j] = phase_half(p[j], j);
    } else {
#pragma unroll
      for (int j = 0; j < S; ++j) p[j] = phase(p[j], j);
    }
    // ---- forward within the warp
    c2 e[S];
    {
      c2 pl = shfl_up2<T>(p[S - 1], 1), pr = shfl_down2<T>(p[0], 1);
      if (lane == 0) pl = w > 0 ? p[0] : zero;             // stand-ins until the exchange
      if (lane == 31) pr = w + 1 < W ? p[S - 1] : zero;
      c2 prev = zero;
#pragma unroll
      for (int j = 0; j < S; ++j) {
        const c2 left = j == 0 ? pl : p[j > 0 ? j - 1 : 0], right = j == S - 1 ? pr : p[j < S - 1 ? j + 1 : j];
        if constexpr (VAR) {
          const c2 lv = mk<T>(lapv(left.x, right.x, p[j].x, hh[j].x, hh[j].y),
                              lapv(left.y, right.y, p[j].y, hh[j].x, hh[j].y));
          const c2 v = cf_mul<T, IMAG>(bf[j], lv);
          prev = j == 0 ? v : cf_fma<T, IMAG>(al[j], prev, v);
        } else {
          const c2 v = j == 0 ? mk<T>(neg_lap(left.x, right.x, p[j].x), neg_lap(left.y, right.y, p[j].y))
                              : mk<T>(lap_add(prev.x, left.x, right.x, p[j].x),
                                      lap_add(prev.y, left.y, right.y, p[j].y));
          prev = cf_mul<T, IMAG>(al[j], v);
        }
        e[j] = prev;
      }
      c2 B = e[S - 1];
#pragma unroll
      for (int l = 0; l < 5; ++l)
        if (l < P.levels) B = cf_fma<T, IMAG>(Pm[l], shfl_up2<T>(B, 1 << l), B);
      if constexpr (S == 1) {
        e[0] = B;
      } else {
        c2 Ein = shfl_up2<T>(B, 1);
        if (lane == 0) Ein = zero;
#pragma unroll
        for (int j = 0; j < S - 1; ++j) e[j] = cf_fma<T, IMAG>(gf[j], Ein, e[j]);
        e[S - 1] = B;
      }
    }
    // ---- first exchange: edge points and the forward end value
    if (C == 1) {
      if (lane == 0) s_first[w] = p[0];
      if (lane == 31) {
        s_last[w] = p[S - 1];
        s_end[w] = e[S - 1];
      }
    } else {
      const c2 f = bcast(p[0], 0), l = bcast(p[S - 1], 31), x = bcast(e[S - 1], 31);
      publish(s_first, w, f);
      publish(s_last, w, l);
      publish(s_end, w, x);
    }
    sync();
    if (w > 0) {
      c2 X = zero, prod = mk<T>(1, 0);
      for (int q = w - 1; q >= 0 && q >= w - P.depth; --q) {
        const c2 f = s_first[q + 1], l = s_last[q], x = s_end[q];
        const c2 d = mk<T>(f.x - l.x, f.y - l.y);
        const c2 g = cf_mul<T, IMAG>(s_cr[q], d);
        const c2 Y = mk<T>(x.x + (d.x - g.x), x.y + (d.y - g.y));
        if (q == w - 1) {
          X = Y;
          prod = s_A[q];
        } else {
          X = cf_fma<T, IMAG>(prod, Y, X);
          prod = cf_cc<T, IMAG>(prod, s_A[q]);
        }
      }
#pragma unroll
      for (int j = 0; j < S; ++j) e[j] = cf_fma<T, IMAG>(gw[j], X, e[j]);
    }
    if (lane == 31 && w + 1 < W) {
      const c2 f = s_first[w + 1];
      const c2 g = cf_mul<T, IMAG>(cr, mk<T>(f.x - p[S - 1].x, f.y - p[S - 1].y));
      e[S - 1] = mk<T>(e[S - 1].x - g.x, e[S - 1].y - g.y);
    }
    // ---- backward within the warp
    {
      c2 next = e[S - 1];
#pragma unroll
      for (int j = S - 2; j >= 0; --j) e[j] = next = cf_fma<T, IMAG>(back(j), next, e[j]);
      // the first point's own value takes its coefficient's product with the
      // thread after: B holds z at the thread's first point
      c2 B = e[0];
#pragma unroll
      for (int l = 0; l < 5; ++l)
        if (l < P.levels) B = cf_fma<T, IMAG>(Qm[l], shfl_down2<T>(B, 1 << l), B);
      if constexpr (S == 1) {
        e[0] = B;
      } else {
        c2 Zin = shfl_down2<T>(B, 1);
        if (lane == 31) Zin = zero;
#pragma unroll
        for (int j = 1; j < S; ++j) e[j] = cf_fma<T, IMAG>(gb[j], Zin, e[j]);
        e[0] = B;
      }
    }
    // ---- second exchange: the warp's first backward value
    if (C == 1) {
      if (lane == 0) s_z[w] = e[0];
    } else {
      publish(s_z, w, bcast(e[0], 0));
    }
    sync();
    {
      c2 Z = s_z[w + 1];
      if (P.depth > 1 && w + 1 < W) {
        c2 prod = s_B[w + 1];
        for (int q = w + 2; q < W && q <= w + P.depth; ++q) {
          Z = cf_fma<T, IMAG>(prod, s_z[q], Z);
          prod = cf_cc<T, IMAG>(prod, s_B[q]);
        }
      }
#pragma unroll
      for (int j = 0; j < S; ++j) p[j] = sub2<T>(p[j], cf_fma<T, IMAG>(gbw[j], Z, e[j]));
    }
    // ---- closing half and norm
    if constexpr (IMAG) {
      if (P.close_each) {
#pragma unroll
        for (int j = 0; j < S; ++j) p[j] = phase(p[j], j);
      }
      NT nval;
      if constexpr (std::is_same<NT, T>::value) {
        nval = T(0);
#pragma unroll
        for (int j = 0; j < S; ++j) nval = nval + wk[j] * (p[j].x * p[j].x + p[j].y * p[j].y);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) nval = nval + shfl_xor_t(nval, o);
      } else {
        nval = NT::zero();
        float m = 0.f;
#pragma unroll
        for (int j = 0; j < S; ++j) m = fmaxf(m, fmaxf(fabsf(p[j].x), fabsf(p[j].y)));
        nval.scale(m);
#pragma unroll
        for (int j = 0; j < S; ++j) {
          nval.square(wk[j], p[j].x);
          nval.square(wk[j], p[j].y);
        }
        nval.warp_total();
      }
      if (C > 1 || lane == 0) publish(s_nrm, w, nval);
      sync();  // third exchange
    }
  }
  if (IMAG) {
    const T scl = line_factor(s_nrm, W, ws);
#pragma unroll
    for (int j = 0; j < S; ++j) {
      p[j].x = p[j].x * scl;
      p[j].y = p[j].y * scl;
    }
  } else if (P.close_end) {
#pragma unroll
    for (int j = 0; j < S; ++j) p[j] = phase_half(p[j], j);
  }
  const long lim = A.geom.points();
#pragma unroll
  for (int j = 0; j < S; ++j)
    if (k0 + j <= M && GPE_CHECK(k0 + j < lim, 291)) A.psi[k0 + j] = p[j];
  if (w == 0 && lane == 0) {
    A.psi[0] = zero;
    A.psi[n - 1] = zero;
  }
}


// Points per thread (S), blocks of the cluster (C) and threads per block for a
// line of M interior points; S = 0: too long for one cluster.  The lines lie
// where the measured step times cross (us per step):
//  * FP32: one block's barriers are cheaper than a cluster's, so a second block
//    only from 512 threads of 4 points on (513 points, imaginary time: 1.58 with
//    one block, 2.02 with four; 1000 real: 1.17 against 1.50; 4001 imaginary,
//    with FP32 norm sums: 2.58 with four blocks of 256 threads, 3.22 with
//    two of 512);
//  * FP64 is bound by its two FP64 lanes per SM and the latency of its chain,
//    so about 64 points per block (256 points: 5.63 with one block, 3.92 with
//    four; 1000: 4.63 with eight, 6.81 with four), and more than one point per
//    thread (fewer warps, each paying the carry arithmetic) only once sixteen
//    blocks are full (4001 real: 9.66, 7.03, 10.18 for S = 1, 2, 4; 8000
//    imaginary: 17.3, 11.8, 9.9);
//  * double-float (at most 514 points): 256 points 3.39 with one block, 4.48
//    with four; 513 points 3.94 and 2.80.
struct LinePlan {
  int S = 0, C = 1, threads = 0;
};

template <typename T>
LinePlan line_plan(int M) {
  LinePlan p;
  if (std::is_same<T, double>::value) {
    p.S = M <= 2048 ? 1 : M <= 6144 ? 2 : 4;
    p.C = M <= 64 ? 1 : M <= 128 ? 2 : M <= 256 ? 4 : M <= 1024 ? 8 : 16;
  } else if (std::is_same<T, float>::value) {
    p.S = M <= 512 ? 1 : 4;
    while (p.C < kLineMaxCtas && M > 4 * (p.C == 1 ? 512 : 256) * p.C) p.C *= 2;
  } else {
    p.S = 1;
    p.C = M <= 256 ? 1 : 4;
  }
  const int per_block = ((M + p.S - 1) / p.S + p.C - 1) / p.C;
  p.threads = (per_block + 31) / 32 * 32;
  if (p.threads > kLineMaxThreads) p.S = 0;
  return p;
}

// Whether the current device can hold a cluster of C blocks of this kernel
// (up to 8 blocks every device can; 16 depend on the device and the block's
// size, and are an attribute of the kernel that each device's context keeps).
template <typename T, bool IMAG, bool VAR, int S>
bool line_fits(int C, int threads) {
  if (C <= 8) return true;
  constexpr int kDevices = 64;
  static std::atomic<signed char> known[kDevices][kLineMaxThreads / 32 + 1] = {};  // 0: not asked; 1: yes; 2: no
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kDevices) return false;
  auto& k = known[dev][threads / 32];
  if (k.load() == 0) {
    auto kern = line_steps_kernel<T, IMAG, VAR, S>;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(C);
    cfg.blockDim = dim3(threads);
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = C;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    int clusters = 0;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveClusters(&clusters, kern, &cfg);
    if (e != cudaSuccess) cudaGetLastError();
    k.store(e == cudaSuccess && clusters > 0 ? 1 : 2);
  }
  return k.load() == 1;
}

template <typename T, bool IMAG, bool VAR, int S>
int launch_line(gp_handle* h, const LineArgs<T>& a, int C, int threads) {
  if (!line_fits<T, IMAG, VAR, S>(C, threads)) return GP_ERR_STATE;
  auto kern = line_steps_kernel<T, IMAG, VAR, S>;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(C);
  cfg.blockDim = dim3(threads);
  cfg.stream = h->work;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = C;
  at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = C > 1 ? 1 : 0;
  GP_CUDA(cudaLaunchKernelEx(&cfg, kern, a));
  count_launch();
  return GP_OK;
}

template <typename T, bool IMAG, bool VAR>
int launch_line_s(gp_handle* h, const LineArgs<T>& a, const LinePlan& p) {
  if constexpr (!is_df<T>::value) {
    if constexpr (std::is_same<T, double>::value)
      if (p.S == 2) return launch_line<T, IMAG, VAR, 2>(h, a, p.C, p.threads);
    if (p.S == 4) return launch_line<T, IMAG, VAR, 4>(h, a, p.C, p.threads);
  }
  return launch_line<T, IMAG, VAR, 1>(h, a, p.C, p.threads);
}

// nsteps steps of a 1d grid (see line_steps_kernel); GP_ERR_STATE if the line
// is too long for one cluster (the caller then steps it launch by launch).
template <typename T>
int run_line_t(gp_handle* h, bool imag, long nsteps) {
  const int mode = imag ? MODE_IMAG : MODE_REAL;
  const LinePlan plan = line_plan<T>(h->n[0] - 2);
  if (plan.S == 0) return GP_ERR_STATE;
  int rc = join_in(h);
  if (rc) return rc;
  const bool merged = h->strang && !imag;  // real-time Strang: the halves between steps merged (StepForm)
  LineArgs<T> L;
  std::memset(&L, 0, sizeof(L));
  auto fill = [&](Sweep2Args<T>& a, bool half) {
    a.psi = (c2_t<T>*)h->psi;
    a.geom = geom_of(h, 0);
    a.alpha = coef_ptr<T>(h, mode, 0, 0);
    set_phase_args<T>(h, imag, half, a);
    a.w_axis = (const T*)h->wt[0];
    a.parts_wscale = h->wscale;
    if (h->geom == 2) {
      const c2_t<T>* cv = (const c2_t<T>*)h->cvar[mode];
      a.vab = cv;
      a.vbf = cv + h->n[0];
      a.vh = cv + 2 * h->n[0];
    }
  };
  fill(L.a, h->strang && imag);
  fill(L.h, h->strang);
  // levels: 2^levels threads of S points reach as far as the coefficients do; depth: the same in warps
  const long reach = h->axis_reach[mode][0];
  while (L.levels < 5 && ((1L << L.levels) - 1) * plan.S < reach) ++L.levels;
  L.depth = (int)std::max<long>(1, std::min<long>(kLineMaxWarps, (reach + 32L * plan.S - 1) / (32L * plan.S)));
  L.close_each = h->strang && imag;
  constexpr long kChunk = 1L << 16;  // steps of one launch
  for (long t = 0; t < nsteps; t += kChunk) {
    L.nsteps = std::min(kChunk, nsteps - t);
    L.half_first = merged && t == 0;
    L.close_end = merged && t + L.nsteps == nsteps;
    if (h->geom == 2)
      rc = imag ? launch_line_s<T, true, true>(h, L, plan) : launch_line_s<T, false, true>(h, L, plan);
    else
      rc = imag ? launch_line_s<T, true, false>(h, L, plan) : launch_line_s<T, false, false>(h, L, plan);
    if (rc) break;  // (GP_ERR_STATE comes from the first launch only: nothing has run)
  }
  const int ro = join_out(h);
  return rc ? rc : ro;
}

}  // namespace gpe
