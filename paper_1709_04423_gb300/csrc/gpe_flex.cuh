// gpe_flex.cuh -- line sweeps on tiles of few lines.
//
// The tile and column sweeps of gpe_sweep2.cuh take 32 lines per block and at
// most 16 segments per line.  That leaves most of the chip idle where a grid
// has few lines (a 2d grid of 257 x 201 points has 7 and 9 such tiles for 152
// SMs), and does not take lines over 514 points.  Here a tile is W lines, W a
// power of two picked so that the tiles fill the SMs (flex_plan), times the
// whole line, staged in shared memory; thread = (line, segment), any number of
// segments per line that the block holds.  Per line the arithmetic is that of
// tsweep_body / colsweep_body with the same segment length (bit for bit, but for
// the sub-step N of FP64 states in imaginary time: from the whole angle here, in
// factor form in tsweep_body, see phase_f64), with more than 16 segments the
// carries' products are formed on the fly from the segment products instead of
// read from the 16 x 16 tables.
//
// Tile layout: line c, point k at c P + k + (k - 1)/SEG (one element skipped
// per segment; see flex_tile).  y/z tiles of W >= 2 (16-byte points) or 4
// (8-byte points) lines move whole 32-byte sectors.
// The coefficients are read through L1 where they are used: staging three
// tables of n points would cost as much as the tile itself for small W.
#pragma once
#include "gpe_sweep2.cuh"

namespace gpe {

constexpr int kFlexMaxThreads = 256;
constexpr int kFlexMinThreads = 128;  // enough threads to bring a small tile in

struct FlexTile {
  int lw;      // log2 W
  int P;       // elements per line in shared memory
  int nseg;    // segments per line
  int depth;   // > 16 segments: segments a carry crosses
};

// The tile of 2^lw lines of n points in segments of seg points.  Its lines
// start P elements apart with P mod U = U/W (U elements fill the 128 bytes of
// one bank row; odd for W >= U): then the W lines and the segments of a warp,
// one bank position apart each, cover every position once.
template <typename T>
__host__ __device__ inline FlexTile flex_tile(int n, int lw, int seg) {
  constexpr int U = 128 / (int)sizeof(c2_t<T>);
  FlexTile t;
  t.lw = lw;
  t.nseg = (n - 2 + seg - 1) / seg;
  const int len = n + t.nseg;
  t.P = (1 << lw) >= U ? len | 1 : (len + U - 1) / U * U + (U >> lw) % U;
  t.depth = 1;
  return t;
}

// Shared memory of a tile, in elements: the lines, then the two carry arrays.
inline size_t flex_elems(const FlexTile& t) { return ((size_t)t.P + 2 * (size_t)t.nseg) << t.lw; }

// The values a solving thread works on: whole complex points, or (SPLIT, FP64
// and double-float) one component each, neighbouring lanes holding the two of a point.  One warp
// gets an FP64 result every 64 clocks whatever its active lanes, four warps
// of an SM together one every 19 (measured with chains of FMAs), so on grids
// with too few lines to keep four warps per SM busy a thread per component
// halves the FP64 instructions of every warp's chain.  Same operations on each
// component, so the same bits.  o: the other component where the caller has
// it at hand (fma_pair), else fetched by a shuffle.
template <typename T, bool IMAG, bool SPLIT>
struct FlexOps {
  using V = c2_t<T>;
  static __device__ __forceinline__ V zero() { return mk<T>(0, 0); }
  static __device__ __forceinline__ V part(const c2_t<T>& p, int) { return p; }
  static __device__ __forceinline__ c2_t<T> full(const V& v, int) { return v; }
  static __device__ __forceinline__ void set(c2_t<T>& d, int, const V& v) { d = v; }
  static __device__ __forceinline__ V other(const V& v) { return v; }
  static __device__ __forceinline__ V lap_add(const V& q, const V& l, const V& r, const V& p) {
    return mk<T>(gpe::lap_add(q.x, l.x, r.x, p.x), gpe::lap_add(q.y, l.y, r.y, p.y));
  }
  static __device__ __forceinline__ V lapv(const V& l, const V& r, const V& p, const c2_t<T>& h) {
    return mk<T>(gpe::lapv(l.x, r.x, p.x, h.x, h.y), gpe::lapv(l.y, r.y, p.y, h.x, h.y));
  }
  static __device__ __forceinline__ V mul(const c2_t<T>& a, const V& b, int) { return cf_mul<T, IMAG>(a, b); }
  static __device__ __forceinline__ V fma(const c2_t<T>& a, const V& b, const V& c, int) {
    return cf_fma<T, IMAG>(a, b, c);
  }
  static __device__ __forceinline__ V fma_pair(const c2_t<T>& a, const V& b, const V&, const V& c, int) {
    return cf_fma<T, IMAG>(a, b, c);
  }
  static __device__ __forceinline__ V sub2(const V& p, const V& z) { return gpe::sub2<T>(p, z); }
  static __device__ __forceinline__ T sq(const V& u) { return u.x * u.x + u.y * u.y; }
};

template <typename T, bool IMAG>
struct FlexOps<T, IMAG, true> {
  using V = T;
  static __device__ __forceinline__ T flip(T v, int comp) { return comp ? v : -v; }  // -v for the real part's thread
  static __device__ __forceinline__ T zero() { return T(0); }
  static __device__ __forceinline__ T part(const c2_t<T>& p, int comp) { return reinterpret_cast<const T*>(&p)[comp]; }
  static __device__ __forceinline__ c2_t<T> full(T v, int comp) {
    const T o = shfl_xor_t(v, 1);
    return comp ? mk<T>(o, v) : mk<T>(v, o);
  }
  static __device__ __forceinline__ void set(c2_t<T>& d, int comp, T v) { reinterpret_cast<T*>(&d)[comp] = v; }
  static __device__ __forceinline__ T other(T v) {
    if constexpr (IMAG) return v;
    else return shfl_xor_t(v, 1);
  }
  static __device__ __forceinline__ T lap_add(T q, T l, T r, T p) { return gpe::lap_add(q, l, r, p); }
  static __device__ __forceinline__ T lapv(T l, T r, T p, const c2_t<T>& h) { return gpe::lapv(l, r, p, h.x, h.y); }
  static __device__ __forceinline__ T mul(const c2_t<T>& a, T b, int comp) {
    if constexpr (IMAG) return a.x * b;
    else if constexpr (is_df<T>::value) return dfl::df_dot2(a.x, b, flip(-a.y, comp), other(b));
    else return ::fma(a.x, b, flip(a.y, comp) * other(b));
  }
  static __device__ __forceinline__ T fma_pair(const c2_t<T>& a, T b, T o, T c, int comp) {
    if constexpr (is_df<T>::value) {
      if constexpr (IMAG) return dfl::fma(a.x, b, c);
      else return dfl::df_dot2_add(a.x, b, flip(-a.y, comp), o, c);
    } else {
      if constexpr (IMAG) return ::fma(a.x, b, c);
      else return ::fma(a.x, b, ::fma(flip(a.y, comp), o, c));
    }
  }
  static __device__ __forceinline__ T fma(const c2_t<T>& a, T b, T c, int comp) {
    return fma_pair(a, b, other(b), c, comp);
  }
  static __device__ __forceinline__ T sub2(T p, T z) {
    if constexpr (is_df<T>::value) return dfl::df_sub2(p, z);
    else return ::fma(T(-2), z, p);
  }
  static __device__ __forceinline__ T sq(T u) { return u * u; }
};

// Lines L0 .. L0 + W - 1 of the grid described by A.  AXIS0: x lines, with
// the sub-step N and the pending factor on the way in (the FIRST of
// tsweep_body); else y/z lines (LAST, CLOSE as colsweep_body).
template <typename T, bool IMAG, bool LAST, int SEG, bool AXIS0, bool VAR, bool CLOSE, bool SPLIT>
__device__ __forceinline__ void flex_body(const Sweep2Args<T>& A, const FlexTile& F, int L0, c2_t<T>* smem,
                                          double* red_smem) {
  static_assert(!AXIS0 || (!LAST && !CLOSE), "x is not the last axis of a 2d/3d grid");
  static_assert(AXIS0 || !VAR, "rho is axis 0");
  using c2 = c2_t<T>;
  constexpr int LS = SEG == 4 ? 2 : SEG == 8 ? 3 : SEG == 16 ? 4 : 5;
  const LineGeom& G = A.geom;
  const int n = G.n, M = n - 2, lw = F.lw, W = 1 << lw;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nwarps = blockDim.x >> 5;
  const int nl = min(W, (int)G.nlines - L0);
  c2* tile = smem;
  c2* cf = smem + ((size_t)F.P << lw);
  c2* cb = cf + (F.nseg << lw);
  auto at = [&](int c, int k) -> c2& { return tile[c * F.P + k + ((k - 1) >> LS)]; };  // 1 <= k <= M
  const c2 zero = mk<T>(0, 0);
  pdl_wait();  // the state and the norm sums are the previous kernels' output
  pdl_release();
  const long lim = G.points();
  // ---- load
  if constexpr (AXIS0) {
    constexpr bool kF64 = std::is_same<T, double>::value;
    const c2* in = A.src ? A.src : A.psi;
    auto apply_N = [&](c2 w, int Lg, int k, T scl) -> c2 {
      const long q = (long)Lg * G.nx + k;
      if constexpr (is_df<T>::value) {
        if (IMAG) { w.x *= scl; w.y *= scl; }
        return phase_df<IMAG>(w, A, q, k, Lg, A.dtg);
      } else {
        w.x *= scl; w.y *= scl;
        const int j = Lg % G.ny, kz = Lg / G.ny;
        const T V = A.V ? A.V[q] : A.vx[k] + (A.vy[j] + A.vz[kz]);
        if constexpr (kF64)
          return phase_f64<IMAG, true>(w, V, A.dt, A.g, [&]() {
            return A.fV ? A.fV[q] : fac_mul<T, IMAG>(A.fx[k], fac_mul<T, IMAG>(A.fy[j], A.fz[kz]));
          });
        else
          return phase_direct<T, IMAG>(w, V, A.dt, A.g);
      }
    };
    const bool pend = A.parts_in != nullptr;
    const int per_line = (n + 31) >> 5, items = nl * per_line;  // 32-point chunks of the tile's rows
    if (pend && warp == 0) {
      const double f = pending_factor_warp(A.parts_in, A.nparts_in, A.parts_wscale);
      if (lane == 0) red_smem[0] = f;
    }
    const int w0 = pend ? 1 : 0;  // first loading warp (a block has at least 4)
    if (warp >= w0)
      for (int i0 = warp - w0; i0 < items; i0 += 4 * (nwarps - w0)) {
        c2 v[4];
#pragma unroll
        for (int r = 0; r < 4; ++r) {
          const int i = i0 + r * (nwarps - w0), c = i / per_line, k = (i - c * per_line) * 32 + lane;
          v[r] = (i < items && k >= 1 && k <= M && GPE_CHECK((long)(L0 + c) * G.nx + k < lim, 301))
                     ? in[(long)(L0 + c) * G.nx + k]
                     : zero;
        }
#pragma unroll
        for (int r = 0; r < 4; ++r) {
          const int i = i0 + r * (nwarps - w0), c = i / per_line, k = (i - c * per_line) * 32 + lane;
          if (i < items && k >= 1 && k <= M) at(c, k) = pend ? v[r] : apply_N(v[r], L0 + c, k, T(1));
        }
      }
    if (pend) {
      __syncthreads();
      const T scl = (T)red_smem[0];
      for (int i = warp; i < items; i += nwarps) {
        const int c = i / per_line, k = (i - c * per_line) * 32 + lane;
        if (k >= 1 && k <= M) at(c, k) = apply_N(at(c, k), L0 + c, k, scl);
      }
    }
  } else {
    const int c = tid & (W - 1), dk = blockDim.x >> lw;
    if (c < nl) {
      const int st = (int)G.stride;
      const long base = line_base(G, L0 + c);
      const c2* line = A.psi + base;
      for (int k0 = 1 + (tid >> lw); k0 <= M; k0 += 8 * dk) {
        c2 v[8];
#pragma unroll
        for (int r = 0; r < 8; ++r) {
          const int k = k0 + r * dk;
          v[r] = (k <= M && GPE_CHECK(base + (long)k * st < lim, 302)) ? line[(long)k * st] : zero;
        }
#pragma unroll
        for (int r = 0; r < 8; ++r) {
          const int k = k0 + r * dk;
          if (k <= M) at(c, k) = v[r];
        }
      }
    }
  }
  __syncthreads();
  // ---- solve: thread = (line c, segment s), or (line, segment, component) with SPLIT
  using X = FlexOps<T, IMAG, SPLIT>;
  using V = typename X::V;
  const int ls = lw + (SPLIT ? 1 : 0);  // log2 of the threads per segment
  const int comp = SPLIT ? tid & 1 : 0;
  const int c = (SPLIT ? tid >> 1 : tid) & (W - 1), s = tid >> ls;
  // whole warps take part (pairs exchange components by shuffles); the last
  // one's threads past the last segment see only points past the line's end
  const bool solving = ((tid & ~31) >> ls) < F.nseg;
  const bool solver = s < F.nseg && c < nl;
  const int k0 = 1 + s * SEG;
  const bool small = F.nseg <= 16;
  const int dep = small ? (A.cdepth > 0 ? A.cdepth : 16) : F.depth;
  const bool whole = k0 + SEG - 1 <= M;
  const c2* bk = VAR ? A.vab : A.alpha;
  V* cfv = reinterpret_cast<V*>(cf);
  V* cbv = reinterpret_cast<V*>(cb);
  auto slot = [&](int q) { return SPLIT ? (((q << lw) + c) << 1) + comp : (q << lw) + c; };
  auto pair_slot = [&](int q) { return SPLIT ? slot(q) ^ 1 : slot(q); };  // the other component's
  // this segment's points in the tile (point k0 + j at seg[j], the two next to it at
  // seg[-2] and seg[SEG + 1]) and how many of them the line has
  c2* seg = tile + c * F.P + k0 + s;
  const int jm = M - k0 + 1;
  auto get = [&](int j) -> V { return X::part(seg[j], comp); };
  const V vzero = X::zero();
  V z[SEG];
#pragma unroll
  for (int j = 0; j < SEG; ++j) z[j] = vzero;  // (unset on one path they would stay live around a caller's loop)
  if (solving) {
    V pm = s > 0 && jm >= 0 ? get(-2) : vzero, pc = jm > 0 ? get(0) : vzero, prev = vzero;
#pragma unroll
    for (int j = 0; j < SEG; ++j) {
      const int k = k0 + j;
      const V pn = j + 1 < jm ? get(j + 1 < SEG ? j + 1 : SEG + 1) : vzero;
      V v = vzero;
      if constexpr (VAR) {
        const c2 h = j < jm ? A.vh[k] : zero;
        const V lv = X::lapv(pm, pn, pc, h);
        v = X::fma(j < jm ? A.alpha[k] : zero, prev, X::mul(j < jm ? A.vbf[k] : zero, lv, comp), comp);
      } else {
        const V t = X::lap_add(prev, pm, pn, pc);
        v = X::mul(j < jm ? A.alpha[k] : zero, t, comp);
      }
      z[j] = v;
      prev = v;
      pm = pc;
      pc = pn;
    }
    V Bend = z[SEG - 1];
#pragma unroll
    for (int j = 0; j < SEG; ++j) if (j + 1 == jm) Bend = z[j];
    if (s < F.nseg) cfv[slot(s)] = Bend;
  }
  __syncthreads();
  if (solving) {
    V Ein = vzero;
    if (small) {
      for (int q = max(0, s - dep); q < s && s < F.nseg; ++q)
        Ein = X::fma_pair(__ldg(&A.ptab[q * 16 + s - 1]), cfv[slot(q)], cfv[pair_slot(q)], Ein, comp);
    } else if (s > 0 && s < F.nseg) {
      Ein = cfv[slot(s - 1)];
      if (dep > 1) {
        c2 prod = __ldg(&A.gf[s * SEG]);  // segment s - 1 ends at point s SEG
        for (int q = s - 2; q >= 0 && q >= s - dep; --q) {
          Ein = X::fma_pair(prod, cfv[slot(q)], cfv[pair_slot(q)], Ein, comp);
          prod = cf_cc<T, IMAG>(prod, __ldg(&A.gf[(q + 1) * SEG]));
        }
      }
    }
    const V Eo = X::other(Ein);
    auto fwd = [&](auto nj) {
#pragma unroll
      for (int j = 0; j < decltype(nj)::value; ++j)
        if (j < jm) z[j] = X::fma_pair(__ldg(&A.gf[k0 + j]), Ein, Eo, z[j], comp);
    };
    if (SEG > 4 && A.cpts == 4) fwd(std::integral_constant<int, (SEG > 4 ? 4 : SEG)>());
    else if (SEG > 8 && A.cpts == 8) fwd(std::integral_constant<int, (SEG > 8 ? 8 : SEG)>());
    else if (SEG > 12 && A.cpts == 12) fwd(std::integral_constant<int, (SEG > 12 ? 12 : SEG)>());
    else fwd(std::integral_constant<int, SEG>());
    V next = vzero;
#pragma unroll
    for (int j = SEG - 1; j >= 0; --j) {
      next = X::fma(j < jm ? bk[k0 + j] : zero, next, z[j], comp);
      if (j >= jm) next = vzero;
      z[j] = next;
    }
    if (s < F.nseg) cbv[slot(s)] = z[0];
  }
  __syncthreads();
  // FP32 states on grids with lines over 514 points (A.norm64): the norm by SquareSum
  constexpr bool kNorm64 = LAST && !CLOSE && std::is_same<T, float>::value;
  T nval = T(0);
  [[maybe_unused]] SquareSum sq = SquareSum::zero();
  if (solving) {
    V Zin = vzero;
    if (small) {
      const int qe = min(F.nseg, s + 1 + dep);
      for (int q = s + 1; q < qe; ++q)
        Zin = X::fma_pair(__ldg(&A.ptab[256 + q * 16 + s + 1]), cbv[slot(q)], cbv[pair_slot(q)], Zin, comp);
    } else if (s + 1 < F.nseg) {
      Zin = cbv[slot(s + 1)];
      if (dep > 1) {
        c2 prod = __ldg(&A.gb[1 + (s + 1) * SEG]);  // segment s + 1 starts there
        for (int q = s + 2; q < F.nseg && q <= s + dep; ++q) {
          Zin = X::fma_pair(prod, cbv[slot(q)], cbv[pair_slot(q)], Zin, comp);
          prod = cf_cc<T, IMAG>(prod, __ldg(&A.gb[1 + q * SEG]));
        }
      }
    }
    const V Zo = X::other(Zin);
    auto bwd = [&](auto nj) {
#pragma unroll
      for (int j = SEG - decltype(nj)::value; j < SEG; ++j)
        if (j < jm) z[j] = X::fma_pair(__ldg(&A.gb[k0 + j]), Zin, Zo, z[j], comp);
    };
    if (SEG > 4 && whole && A.cpts == 4) bwd(std::integral_constant<int, (SEG > 4 ? 4 : SEG)>());
    else if (SEG > 8 && whole && A.cpts == 8) bwd(std::integral_constant<int, (SEG > 8 ? 8 : SEG)>());
    else if (SEG > 12 && whole && A.cpts == 12) bwd(std::integral_constant<int, (SEG > 12 ? 12 : SEG)>());
    else bwd(std::integral_constant<int, SEG>());
    // ---- u = p - 2 z: x tiles back into shared memory, y/z lines stored from here
    if constexpr (AXIS0) {
#pragma unroll
      for (int j = 0; j < SEG; ++j)
        if (j < jm && solver) X::set(seg[j], comp, X::sub2(get(j), z[j]));
    } else {
      const int L = L0 + c, st = (int)G.stride;
      const long base = solver ? line_base(G, L) : 0;
      c2* line = A.psi + base;
      const int ci = L % G.nx, cf2 = L / G.nx;
      T tacc = T(0);
#pragma unroll
      for (int j = 0; j < SEG; ++j) {
        const int k = k0 + j;
        V u = j < jm ? X::sub2(get(j), z[j]) : vzero;
        if constexpr (CLOSE) {
          c2 f = X::full(u, comp);
          if (j < jm && solver)
            f = half_phase<T, IMAG>(A, f, base + (long)k * st, ci, G.axis == 2 ? cf2 : k, G.axis == 2 ? k : cf2);
          u = X::part(f, comp);
        }
        if (j < jm && solver) {
          if (GPE_CHECK(base + (long)k * st < lim, 303)) X::set(line[(long)k * st], comp, u);
          if (LAST && !(kNorm64 && A.norm64)) tacc += A.w_axis[k] * X::sq(u);
        }
        if constexpr (kNorm64) z[j] = u;
      }
      if constexpr (kNorm64) {
        if (A.norm64) {
          float m = 0.f;
          if (solver)
#pragma unroll
            for (int j = 0; j < SEG; ++j) m = fmaxf(m, fmaxf(fabsf(z[j].x), fabsf(z[j].y)));  // (zeros past the line)
          sq.scale(m);
          if (solver) {
            const float wl = A.w_a[ci] * A.w_b[cf2];
#pragma unroll
            for (int j = 0; j < SEG; ++j) {
              const float w = j < jm ? A.w_axis[k0 + j] * wl : 0.f;
              sq.square(w, z[j].x);
              sq.square(w, z[j].y);
            }
          }
          sq.warp_total();
        }
      }
      if (s == 0 && solver && GPE_CHECK(base + (long)(n - 1) * st < lim, 304)) {
        X::set(line[0], comp, vzero);
        X::set(line[(long)(n - 1) * st], comp, vzero);
      }
      if (LAST && solver) nval = tacc * (A.w_a[ci] * A.w_b[cf2]);
    }
  }
  if constexpr (AXIS0) {
    __syncthreads();
    const int per_line = (n + 31) >> 5, items = nl * per_line;
    for (int i = warp; i < items; i += nwarps) {
      const int cc = i / per_line, k = (i - cc * per_line) * 32 + lane;
      if (k < n && GPE_CHECK((long)(L0 + cc) * G.nx + k < lim, 305))
        A.psi[(long)(L0 + cc) * G.nx + k] = (k >= 1 && k <= M) ? at(cc, k) : zero;
    }
  }
  if constexpr (kNorm64) {
    if (A.norm64) {
      __shared__ SquareSum s_sq[kFlexMaxThreads / 32];
      if (lane == 0) s_sq[warp] = sq;
      __syncthreads();
      if (warp == 0) {
        sq = SquareSum::gather(s_sq, nwarps);
        if (lane == 0) A.parts_out[blockIdx.x] = sq.value();
      }
      return;
    }
  }
  finish_norm<T, LAST>(nval, A.parts_out);
}

template <typename T, bool IMAG, bool LAST, int SEG, bool AXIS0, bool VAR, bool CLOSE, bool SPLIT>
__global__ void __launch_bounds__(kFlexMaxThreads) flex_kernel(const __grid_constant__ Sweep2Args<T> A,
                                                               const __grid_constant__ FlexTile F) {
  extern __shared__ __align__(16) unsigned char fsmem_raw[];
  __shared__ double red_smem[32];
  flex_body<T, IMAG, LAST, SEG, AXIS0, VAR, CLOSE, SPLIT>(A, F, blockIdx.x << F.lw,
                                                          reinterpret_cast<c2_t<T>*>(fsmem_raw), red_smem);
}

// The norm sums of a sweep that left many (more than a warp of every block of
// the next step should add up) as one.
static __global__ void __launch_bounds__(1024) fold_parts_kernel(double* parts, int nparts) {
  __shared__ double smem[32];
  pdl_wait();
  pdl_release();
  double v[1] = {0.0};
  for (int b = threadIdx.x; b < nparts; b += blockDim.x) v[0] += __ldcg(&parts[b]);
  block_sum<1>(v, smem);
  __syncthreads();
  if (threadIdx.x == 0) parts[0] = v[0];
}

// W, segment length and threads of a sweep of nlines lines of n points, or
// threads = 0 where it does not fit a block.  seg: the handle's segment length
// where the sweep must keep its bits (every tile width does), 0: free.
struct FlexPlan {
  FlexTile t = {0, 0, 0, 0};
  int seg = 0, threads = 0;
  unsigned blocks = 0;
  bool split = false;  // FP64 and double-float: a thread per component
};

// The tile is the widest of 16 lines and fewer that gives one and a half
// blocks per SM.  Where the solving warps would still be fewer than four per SM
// (an SM's FP64 rate needs four; the other chains only get shorter), free segments
// are halved down to 8 points and FP64 and double-float take a thread per
// component -- unless the line then needs more threads than a block has (over
// 4098 points), which leaves both components to one thread: 5000 x 50 FP64
// imaginary time 111 us per step, with a thread per line 8870.
template <typename T>
FlexPlan flex_plan(int n, long nlines, int seg, bool axis0, long reach) {
  FlexPlan p;
  const int M = n - 2;
  const int lmin = axis0 ? 1 : sizeof(c2_t<T>) == 8 ? 2 : 1;
  const bool few = nlines * ((M + 15) / 16) < 32L * 4 * 152;
  p.split = few && !std::is_same<T, float>::value;
  for (;; p.split = false) {
    for (int lw = 4; lw >= 0; --lw) {
      const int ls = lw + (p.split ? 1 : 0);
      p.seg = seg;
      if (seg == 0)
        for (int sg : {8, 16, 32}) {
          if (sg == 8 && !few) continue;
          p.seg = sg;
          if ((((M + sg - 1) / sg) << ls) <= kFlexMaxThreads) break;
        }
      p.t = flex_tile<T>(n, lw, p.seg);
      p.t.depth = (int)std::max<long>(1, (reach + p.seg - 1) / p.seg);
      p.threads = std::max(kFlexMinThreads, ((p.t.nseg << ls) + 31) / 32 * 32);
      p.blocks = (unsigned)((nlines + (1L << lw) - 1) >> lw);
      const bool fits = p.threads <= kFlexMaxThreads && flex_elems(p.t) * sizeof(c2_t<T>) <= 200 * 1024;
      if (fits && (lw <= lmin || p.blocks >= 228)) return p;
    }
    if (!p.split) return FlexPlan();
  }
}

template <typename T, bool IMAG, bool LAST, int SEG, bool AXIS0, bool VAR, bool CLOSE>
void launch_flex(const Sweep2Args<T>& a, const FlexPlan& p, cudaStream_t s, bool pdl) {
  auto kern = flex_kernel<T, IMAG, LAST, SEG, AXIS0, VAR, CLOSE, false>;
  if constexpr (!std::is_same<T, float>::value)
    if (p.split) kern = flex_kernel<T, IMAG, LAST, SEG, AXIS0, VAR, CLOSE, true>;
  opt_in_smem((const void*)kern, 200 * 1024);
  launch_k(pdl, kern, dim3(p.blocks), dim3(p.threads), flex_elems(p.t) * sizeof(c2_t<T>), s, a, p.t);
}

template <typename T, bool IMAG, bool LAST, bool AXIS0, bool VAR, bool CLOSE>
void launch_flex_seg(const Sweep2Args<T>& a, const FlexPlan& p, cudaStream_t s, bool pdl) {
  switch (p.seg) {
    case 4: return launch_flex<T, IMAG, LAST, 4, AXIS0, VAR, CLOSE>(a, p, s, pdl);
    case 8: return launch_flex<T, IMAG, LAST, 8, AXIS0, VAR, CLOSE>(a, p, s, pdl);
    case 16: return launch_flex<T, IMAG, LAST, 16, AXIS0, VAR, CLOSE>(a, p, s, pdl);
    default: return launch_flex<T, IMAG, LAST, 32, AXIS0, VAR, CLOSE>(a, p, s, pdl);
  }
}

// One x sweep (with N; var: the rho axis) or y/z sweep (last: with the norm;
// close: after the closing half) with the plan's tiles; instantiated once per
// precision (gpe_flex_*.cu).
template <typename T>
void run_flex(const Sweep2Args<T>& a, const FlexPlan& p, bool imag, bool last, bool close, bool var, cudaStream_t s,
              bool pdl);

template <>
void run_flex<float>(const Sweep2Args<float>&, const FlexPlan&, bool, bool, bool, bool, cudaStream_t, bool);
template <>
void run_flex<double>(const Sweep2Args<double>&, const FlexPlan&, bool, bool, bool, bool, cudaStream_t, bool);
template <>
void run_flex<df64>(const Sweep2Args<df64>&, const FlexPlan&, bool, bool, bool, bool, cudaStream_t, bool);

template <typename T>
void run_flex_t(const Sweep2Args<T>& a, const FlexPlan& p, bool imag, bool last, bool close, bool var, cudaStream_t s,
                bool pdl) {
  if (a.geom.axis == 0) {
    if (var)
      imag ? launch_flex_seg<T, true, false, true, true, false>(a, p, s, pdl)
           : launch_flex_seg<T, false, false, true, true, false>(a, p, s, pdl);
    else
      imag ? launch_flex_seg<T, true, false, true, false, false>(a, p, s, pdl)
           : launch_flex_seg<T, false, false, true, false, false>(a, p, s, pdl);
  } else if (!imag) {
    launch_flex_seg<T, false, false, false, false, false>(a, p, s, pdl);
  } else if (close) {
    launch_flex_seg<T, true, true, false, false, true>(a, p, s, pdl);
  } else if (last) {
    launch_flex_seg<T, true, true, false, false, false>(a, p, s, pdl);
  } else {
    launch_flex_seg<T, true, false, false, false, false>(a, p, s, pdl);
  }
}

}  // namespace gpe
