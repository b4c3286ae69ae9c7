// Traces in the eigenbasis of the blocks (internal; instantiated per precision in kt_eig_*.cu).
//
// H_loc is block diagonal with blocks of at most 36 rows on this path, and setup diagonalises
// every block. A state is carried as its components on the eigenvectors of its block: an
// interval multiplies component k by exp(-dt (lambda_k - lambda_0)), and c_f or c_f^+ is the
// dense matrix V_target^T P V_source between two blocks' eigenvectors, which kt_model_create
// forms once on the device. One operator with the interval after it is then one small
// matrix-vector product and one exponential per component, where the Krylov propagation of
// kt_items.cuh runs two to ten Lanczos steps and the eigensolve of T_p: about 50 dependent warp
// instructions per operator against 2,300.
//
// What bounds it: the serial chain of a walker's operators (matrix-vector product, shared
// memory exchange, exponential), about 85 long per half for the longest walkers of the
// five-orbital batch; no pipe and no memory level is near its limit.
#pragma once

#include <algorithm>
#include <type_traits>

#include "kt_device.cuh"

namespace kt {
namespace dev {

// How a unit's vector is held. EIG_F64: FP64. EIG_PAIR, the FP32 path: a component x is a pair of
// floats, x = h + l with h a multiple of 2^-10 and |l| <= 2^-11, and a matrix entry a pair with h
// a multiple of 2^-11. The vector's norm stays below 8, so the products h h and their sums over a
// row are exact in FP32, and the three other products are summed in FP32 where they are 2^-11
// smaller: an absolute error near 2^-34 for four FMAs a term. That is 33 bits of a vector of size 1,
// 30 of one whose largest component is 1/16 (below it the next interval scales by 16) and 26 at 2^-8,
// where it is scaled at once. A cached state is rounded to one float per component: errors of cached
// log-ratios 3.2e-8 rms, 1.3e-7 at most at five orbitals (4,096 walkers), against 1.7e-9 and 1.7e-8
// from scratch. Plain FP32 components throughout had an error of 4.7e-7 rms in log|T| at five
// orbitals, but up to 1.7e-5 where a trace cancels and 2.5e-5 at seven orbitals; pairs with TwoSum
// sums (12 operations a term) gave no smaller errors that a float could show.
constexpr int EIG_PAIR = 0, EIG_F64 = 1;

template <int MODE>
struct EigT;
template <>
struct EigT<EIG_PAIR> {
  using E = float2;
  static constexpr int EPV = 2;  // elements per 16-byte vector
};
template <>
struct EigT<EIG_F64> {
  using E = double;
  static constexpr int EPV = 2;
};

__device__ __forceinline__ void eig_two_sum(float a, float b, float &s, float &e) {
  s = a + b;
  const float bb = s - a;
  e = (a - (s - bb)) + (b - bb);
}

// (n_up, n_dn) travel as n_up + 1024 n_dn. Block of a (n_up, n_dn, singly-occupied mask) key, -1
// if there is none; kt_model_create checks that c_f and c_f^+ reach a block exactly when the
// moved key has one.
__device__ __forceinline__ int key_block(const DevModel &M, int nn, int mask) {
  const int nu = nn & 1023, nd = nn >> 10;
  if ((unsigned)nu > (unsigned)M.n_orb || (unsigned)nd > (unsigned)M.n_orb) return -1;
  return __ldg(M.key_lut + (((nu * (M.n_orb + 1) + nd) << M.n_orb) | mask));
}

// Change of the key by an operator (code = 2 f + dag).
__device__ __forceinline__ int key_step(int code) {
  return ((code & 1) ? 1 : -1) * ((code & 2) ? 1024 : 1);
}
// Inclusive prefix over the G lanes of a group: sums of nn, exclusive-ors of mk. (Shuffles take a
// third of the instructions of counting ballots per spin and orbital.)
template <int G>
__device__ __forceinline__ void key_scan(int &nn, int &mk, int gl) {
#pragma unroll
  for (int o = 1; o < G; o <<= 1) {
    const int a = __shfl_up_sync(FULL, nn, o, G), b = __shfl_up_sync(FULL, mk, o, G);
    if (gl >= o) {
      nn += a;
      mk ^= b;
    }
  }
}

// ---------------------------------------------------------------------------
// 2^(-dt lambda2) of one component, lambda2 = (lambda_k - lambda_0) log2 e: reduction to the nearest entry
// of a table of powers of two and a Taylor series of the rest (the table-driven method of P. T. P. Tang,
// ACM Trans. Math. Softw. 15, 1989)
// ---------------------------------------------------------------------------
struct EigDt {
  float h, l;   // EIG_PAIR: dt as a pair
  double d;     // EIG_F64
};

// Pairs: 2^-x = 2^k 2^(j/32) e^r with |r| <= ln2/64; table of 2^(j/32) as pairs, the Taylor
// series of e^r to fourth order (fifth-order term below 2e-12).
__device__ __forceinline__ float2 eig_weight_pair(float2 lam, const EigDt &dt, const float2 *__restrict__ tab) {
  const float xh = dt.h * lam.x;
  if (!(xh < 125.f)) return make_float2(0.f, 0.f);
  float xl = fmaf(dt.h, lam.x, -xh);
  xl = fmaf(dt.h, lam.y, xl);
  xl = fmaf(dt.l, lam.x, xl);
  const float t = fmaf(xh, -32.f, 12582912.f);  // 1.5 * 2^23: rounded to an integer in the low bits
  const int i = __float_as_int(t) - 0x4b400000;
  const float f = fmaf(t - 12582912.f, -0.03125f, -xh);  // exact
  const float L2H = 0.693147182f, L2L = -1.90465421e-9f;  // ln 2 as a pair
  const float rh = f * L2H;
  float rl = fmaf(f, L2H, -rh);
  rl = fmaf(f, L2L, rl);
  rl = fmaf(-xl, L2H, rl);
  const float q = rh * rh * fmaf(rh, fmaf(rh, 0.0416666667f, 0.166666667f), 0.5f);
  const float c = rl + q;
  const float s = rh + c, sl = c - (s - rh);
  const float2 T = __ldg(tab + (i & 31));
  const float ph = T.x * s;
  float pl = fmaf(T.x, s, -ph);
  pl = fmaf(T.x, sl, pl);
  pl = fmaf(T.y, s, pl) + T.y;
  const float hi = T.x + ph;
  const float lo = (ph - (hi - T.x)) + pl;
  const float sc = __int_as_float(((i >> 5) + 127) << 23);  // 2^k, k >= -126
  const float rhi = hi + lo;
  return make_float2(rhi * sc, (lo - (rhi - hi)) * sc);
}

// FP64: 2^-x = 2^k 2^(j/128) e^r with |r| <= ln2/256, Taylor series to fifth order (sixth-order
// term 6e-19). A third fewer FP64 instructions than exp(): the FP64 pipe issues one warp
// instruction per 16 cycles.
__device__ __forceinline__ double eig_weight_f64(double lam, double dt, const double *__restrict__ tab) {
  const double x = dt * lam;
  if (!(x < 1000.0)) return 0.0;
  const double magic = 6755399441055744.0;  // 1.5 * 2^52
  const double t = fma(x, -128.0, magic);
  const int i = __double2loint(t);
  const double f = fma(t - magic, -0.0078125, -x);  // exact
  const double r = f * 0.693147180559945309417;
  double p = fma(r, 1.0 / 120.0, 1.0 / 24.0);
  p = fma(r, p, 1.0 / 6.0);
  p = fma(r, p, 0.5);
  p = fma(r * r, p, r);
  const double T = __ldg(tab + (i & 127));
  const double v = fma(T, p, T);  // in [1, 2)
  return __hiloint2double(__double2hiint(v) + ((i >> 7) << 20), __double2loint(v));  // k >= -1000
}

// ---------------------------------------------------------------------------
// One half of an item on one lane group
// ---------------------------------------------------------------------------
template <int MODE, int G, int DMAX>
struct EigHalf {
  using T = EigT<MODE>;
  using E = typename T::E;
  static constexpr int DP = (DMAX + 3) / 4 * 4;  // padded rows of a vector in shared memory
  static constexpr int R = (DP + G - 1) / G;     // rows per lane
  static constexpr int NV = DP / T::EPV;
  E x[R];      // rows gl + G j of the current vector
  double L;    // log-weight (complete after finish())
  int b;       // block
  int dim;
  bool vanished;
};

template <int MODE>
__device__ __forceinline__ typename EigT<MODE>::E eig_zero() {
  if constexpr (MODE == EIG_PAIR) return make_float2(0.f, 0.f);
  else return 0;
}
template <int MODE>
__device__ __forceinline__ typename EigT<MODE>::E eig_one() {
  if constexpr (MODE == EIG_PAIR) return make_float2(1.f, 0.f);
  else return 1;
}
template <int MODE>
__device__ __forceinline__ double eig_value(typename EigT<MODE>::E v) {
  if constexpr (MODE == EIG_PAIR) return (double)v.x + (double)v.y;
  else return (double)v;
}
// hi + lo (|lo| <= ulp(hi) / 2, |hi| < 8) with the first part on the grid of EIG_PAIR
__device__ __forceinline__ float2 eig_split(float hi, float lo) {
  const float h = (hi + 12288.f) - 12288.f;  // 1.5 * 2^13: the sum's last bit is 2^-10
  return make_float2(h, (hi - h) + lo);
}
template <int MODE>
__device__ __forceinline__ typename EigT<MODE>::E eig_from(double a) {
  if constexpr (MODE == EIG_PAIR) {
    const float h = (float)a;
    return eig_split(h, (float)(a - (double)h));
  } else {
    return a;
  }
}
template <int MODE>
__device__ __forceinline__ bool eig_nonzero(typename EigT<MODE>::E v) {
  if constexpr (MODE == EIG_PAIR) return v.x != 0.f || v.y != 0.f;
  else return v != 0;
}
// |v| is large enough that the vector needs no rescaling yet
template <int MODE>
__device__ __forceinline__ bool eig_large(typename EigT<MODE>::E v) {
  if constexpr (MODE == EIG_PAIR) return fabsf(v.x) >= 0.00390625f;
  else return (__double2hiint(v) & 0x7fffffff) >= 0x22d00000;  // 2^-466, without the FP64 pipe
}
template <int MODE>
__device__ __forceinline__ int eig_exponent(typename EigT<MODE>::E v) {  // of a nonzero finite value
  if constexpr (MODE == EIG_PAIR) return ilogbf(v.x);
  else return ilogb(v);
}
template <int MODE>
__device__ __forceinline__ typename EigT<MODE>::E eig_scale(typename EigT<MODE>::E v, int e) {
  if constexpr (MODE == EIG_PAIR) return make_float2(scalbnf(v.x, e), scalbnf(v.y, e));
  else return scalbn(v, e);
}
__device__ __forceinline__ float2 eig_mul_pair(float2 x, float2 w) {
  const float p = x.x * w.x;
  float pe = fmaf(x.x, w.x, -p);
  pe = fmaf(x.x, w.y, pe);
  pe = fmaf(x.y, w.x, pe);
  const float h = p + pe;
  return make_float2(h, pe - (h - p));
}

template <int MODE>
__device__ __forceinline__ typename EigT<MODE>::E eig_lambda(const DevModel &M, int at) {
  return __ldg((const typename EigT<MODE>::E *)M.eig_lam + at);
}
template <int MODE>
__device__ __forceinline__ typename EigT<MODE>::E eig_weight(const DevModel &M, typename EigT<MODE>::E lam, const EigDt &dt) {
  if constexpr (MODE == EIG_PAIR) return eig_weight_pair(lam, dt, (const float2 *)M.eig_tab);
  else return eig_weight_f64(lam, dt.d, (const double *)M.eig_tab);
}

// x (EIG_PAIR: any pair) times the weights wt of an interval dt in the block whose first
// eigenvalue is at eoff. The weights are relative to the block's lowest eigenvalue. When that
// leaves every component small (a vector without components on the low eigenvalues, or a
// small matrix element), the weights are formed again relative to the lowest eigenvalue that
// the vector holds and the vector is rescaled by a power of two; both go to the log-weight.
// EIG_PAIR: a vector whose components fall below 1/16 is scaled by 16 in the next interval (sc),
// which costs no reduction and no wait. False if the vector is exactly zero. `act`: the group
// has such an interval (the others keep x); all lanes of the warp call it together.
template <int MODE, int G, int R>
__device__ __forceinline__ bool eig_interval(const DevModel &M, typename EigT<MODE>::E (&x)[R],
                                             const typename EigT<MODE>::E (&wt)[R], bool act, int gl, int eoff, int d,
                                             const EigDt &dt, double &Lx, int &ex, float &sc) {
  using E = typename EigT<MODE>::E;
  E y[R];
  bool large = false, big = false;
#pragma unroll
  for (int j = 0; j < R; ++j) {
    const int r = gl + G * j;
    y[j] = eig_zero<MODE>();
    if (r < d) {
      if constexpr (MODE == EIG_PAIR) {
        y[j] = eig_mul_pair(x[j], make_float2(wt[j].x * sc, wt[j].y * sc));
        big |= fabsf(y[j].x) >= 0.0625f;
      } else {
        y[j] = x[j] * wt[j];
      }
    }
    large |= eig_large<MODE>(y[j]);
  }
  const unsigned bal = __ballot_sync(FULL, large);
  const unsigned gm = G == 32 ? FULL : (((1u << (G & 31)) - 1u) << ((threadIdx.x & 31) / G * G));
  const bool low = act && !(bal & gm);
  float sn = 1.f;
  if constexpr (MODE == EIG_PAIR) {
    if (act && sc != 1.f) ex -= 4;
    sn = (__ballot_sync(FULL, big) & gm) ? 1.f : 16.f;
  }
  bool alive = true;
  if (__any_sync(FULL, low)) {
    if (MODE == EIG_PAIR && low && sc != 1.f) ex += 4;  // the vector is formed again from x
    int kmin = 1 << 20;
#pragma unroll
    for (int j = R - 1; j >= 0; --j)
      if (gl + G * j < d && eig_nonzero<MODE>(x[j])) kmin = gl + G * j;
#pragma unroll
    for (int o = G / 2; o > 0; o >>= 1) kmin = min(kmin, __shfl_xor_sync(FULL, kmin, o));
    if (kmin >= (1 << 20)) {
      alive = !low;
      kmin = 0;
    }
    const double l0 = __ldg(M.st_eval64 + eoff + (low ? kmin : 0));
    E z[R];
    int e = -100000;
#pragma unroll
    for (int j = 0; j < R; ++j) {
      const int r = gl + G * j;
      z[j] = eig_zero<MODE>();
      if (low && r < d && eig_nonzero<MODE>(x[j])) {
        if constexpr (MODE == EIG_F64) {
          const double lam = __ldg((const double *)M.eig_lam + eoff + r) - __ldg((const double *)M.eig_lam + eoff + kmin);
          z[j] = x[j] * eig_weight_f64(lam, dt.d, (const double *)M.eig_tab);
          if (z[j] != 0.0) e = max(e, eig_exponent<MODE>(z[j]));
        } else {
          const float2 a = __ldg((const float2 *)M.eig_lam + eoff + r), c = __ldg((const float2 *)M.eig_lam + eoff + kmin);
          float s, t;
          eig_two_sum(a.x, -c.x, s, t);
          t += a.y - c.y;
          const float2 lam = make_float2(s + t, t - ((s + t) - s));
          z[j] = eig_mul_pair(x[j], eig_weight_pair(lam, dt, (const float2 *)M.eig_tab));
          if (z[j].x != 0.f) e = max(e, eig_exponent<MODE>(z[j]));
        }
      }
    }
#pragma unroll
    for (int o = G / 2; o > 0; o >>= 1) e = max(e, __shfl_xor_sync(FULL, e, o));
    if (low && e == -100000) alive = false;
    if (low && alive) {
#pragma unroll
      for (int j = 0; j < R; ++j) y[j] = eig_scale<MODE>(z[j], -e);
      ex += e;
      Lx -= (MODE == EIG_F64 ? dt.d : (double)dt.h + (double)dt.l) * l0;
      sn = 1.f;
    }
  }
  if (act) {
    sc = sn;
#pragma unroll
    for (int j = 0; j < R; ++j) {
      if constexpr (MODE == EIG_PAIR) x[j] = eig_split(y[j].x, y[j].y);
      else x[j] = y[j];
    }
  }
  return alive;
}

// One 16-byte vector of a row (two entries) times the vector in shared memory, EIG_PAIR, blocks of at most
// 12 rows. a[0] collects the exact products of the first parts; the three small products have sums of
// their own, chains of two FMAs a vector where eig_fma's one sum makes a chain of six.
__device__ __forceinline__ void eig_fma4(float (&a)[4], const float4 &m, const float4 &v) {
  a[0] = fmaf(m.x, v.x, a[0]);
  a[1] = fmaf(m.x, v.y, a[1]);
  a[2] = fmaf(m.y, v.x, a[2]);
  a[3] = fmaf(m.y, v.y, a[3]);
  a[0] = fmaf(m.z, v.z, a[0]);
  a[1] = fmaf(m.z, v.w, a[1]);
  a[2] = fmaf(m.w, v.z, a[2]);
  a[3] = fmaf(m.w, v.w, a[3]);
}

// One 16-byte vector of a row of an operator matrix (two entries) times the vector in shared
// memory. EIG_PAIR: acc.x collects the exact products of the first parts, acc.y the others.
template <int MODE>
__device__ __forceinline__ void eig_fma(typename EigT<MODE>::E &acc, const float4 &m, const float4 &v) {
  if constexpr (MODE == EIG_PAIR) {
    acc.x = fmaf(m.x, v.x, acc.x);
    acc.y = fmaf(m.x, v.y, acc.y);
    acc.y = fmaf(m.y, v.x, acc.y);
    acc.y = fmaf(m.y, v.y, acc.y);
    acc.x = fmaf(m.z, v.z, acc.x);
    acc.y = fmaf(m.z, v.w, acc.y);
    acc.y = fmaf(m.w, v.z, acc.y);
    acc.y = fmaf(m.w, v.w, acc.y);
  } else {
    const double2 md = *reinterpret_cast<const double2 *>(&m), vd = *reinterpret_cast<const double2 *>(&v);
    acc = fma(md.x, vd.x, acc);
    acc = fma(md.y, vd.y, acc);
  }
}

// Operators at equal times (code = 2 f + dag, from block bs to bt): between them the vector stays
// in the occupation basis, where c_f and c_f^+ are gathers and exact zeros stay exact.
// xs[cb] holds the vector (components, or rows when `fock`); the result's rows go to xs[cb] and
// its components to xs[cb ^ 1]. `on`: the group has such an operator; all lanes of the warp call
// it together. Continuous times never coincide, so this is kept small, in FP64.
template <int MODE, int G, int DMAX>
__device__ __forceinline__ void eig_tied(const DevModel &M, typename EigT<MODE>::E *xs, int cb, bool on, bool fock, int bs,
                                      int bt, int code) {
  using H = EigHalf<MODE, G, DMAX>;
  using E = typename EigT<MODE>::E;
  constexpr int R = H::R, DP = H::DP;
  const int gl = (threadIdx.x & 31) % G;
  const int ds = __ldg(M.blk_dim + bs), dt = __ldg(M.blk_dim + bt), off = __ldg(M.blk_off + bt);
  E *cur = xs + cb * DP, *oth = xs + (cb ^ 1) * DP;
#pragma unroll
  for (int j = 0; j < R; ++j) {
    const int r = gl + G * j;
    if (on && r < ds) {
      E e = cur[r];
      if (!fock) {
        const double *V = M.blk_evec64 + __ldg(M.blk_evoff + bs);
        double a = 0.0;
        for (int k = 0; k < ds; ++k) a = fma(__ldg(V + k * ds + r), eig_value<MODE>(cur[k]), a);
        e = eig_from<MODE>(a);
      }
      oth[r] = e;
    }
  }
  __syncwarp();
  E v[R];
#pragma unroll
  for (int j = 0; j < R; ++j) {
    const int r = gl + G * j;
    v[j] = eig_zero<MODE>();
    if (on && r < dt && ((__ldg(M.st_bits + off + r) >> (code >> 1)) & 1) == (code & 1)) {
      const unsigned pe = __ldg(M.partner + (size_t)(off + r) * M.nf + (code >> 1));
      v[j] = oth[pe & 0x7fffu];
      if (pe & 0x8000u) {
        if constexpr (MODE == EIG_PAIR) v[j] = make_float2(-v[j].x, -v[j].y);
        else v[j] = -v[j];
      }
    }
  }
#pragma unroll
  for (int j = 0; j < R; ++j) {
    const int r = gl + G * j;
    if (on && r < DP) cur[r] = v[j];
  }
  __syncwarp();
#pragma unroll
  for (int j = 0; j < R; ++j) {
    const int k = gl + G * j;
    if (on && k < DP) {
      const double *V = M.blk_evec64 + __ldg(M.blk_evoff + bt) + (size_t)k * dt;
      double a = 0.0;
      if (k < dt)
        for (int r = 0; r < dt; ++r) a = fma(__ldg(V + r), eig_value<MODE>(cur[r]), a);
      oth[k] = eig_from<MODE>(a);
    }
  }
  __syncwarp();
}

// One half of an item: `n` operators from index i0 on, upwards (half 0) or their adjoints
// downwards (half 1), each followed by the interval to the next one and the last by the interval
// to t_end. It starts from kept state q at tau = 0 or beta, or (entry >= 0) from a cached state at
// time t0. n < 0: the group has no item.
struct EigWork {
  int i0, n, half, q;
  double t_end;
  // cached halves: the state to start from, and where the states passed go
  long long entry;   // cache entry of the start state, -1: the kept state
  double t0;         // its time
  size_t eb;         // first entry of the item
  int lo, hi;        // states of positions up to lo (forward), from hi on (backward) go to the cache
                     // itself, the others to the scratch arrays
  bool store;
};

// The lanes of a group take one operator each of the next G (its block from the key prefixes,
// its matrix, its interval), then the group walks through them. Every group of the warp makes
// the same number of turns, so that all warp primitives are converged. CACHED: halves that start
// from or store to the partial-state cache. Their block path may break, in a BUILD because it covers items
// that pruning would remove, else because the caller's sequences are not the cached ones: the states from
// there on are zero.
template <int MODE, int G, int DMAX, bool CACHED, bool BUILD>
__device__ __forceinline__ void eig_half(const DevModel &M, const Cursor &cur, int Kn, const EigWork &wk,
                                         const CacheView &C, typename EigT<MODE>::E *xs, EigHalf<MODE, G, DMAX> &u) {
  using H = EigHalf<MODE, G, DMAX>;
  using T = EigT<MODE>;
  using E = typename T::E;
  using V = typename std::conditional<MODE == EIG_F64, double, float>::type;  // element of a cache entry
  constexpr int R = H::R, DP = H::DP, NV = H::NV;
  const int lane = threadIdx.x & 31, gl = lane % G, half = wk.half;
  const bool on = wk.n >= 0;
  int n = on ? wk.n : 0;
  const double tf = n > 0 ? cur.get(wk.i0).t : wk.t_end;  // end of the interval before the first operator
  double L0 = 0.0, Lx = 0.0;
  int ex = 0;
  float sc = 1.f;
  u.vanished = false;
  if (!CACHED || wk.entry < 0) {
    // the kept state is an eigenvector: a unit vector, and a scalar up to the first operator
    u.b = on ? __ldg(M.kept_blk + wk.q) : 0;
    const int kr = on ? __ldg(M.kept_row + wk.q) : 0;
    const double Ek = on ? __ldg(M.kept_e + wk.q) : 0.0;
    L0 = half ? -(M.beta - tf) * Ek : -tf * Ek;
#pragma unroll
    for (int j = 0; j < R; ++j) u.x[j] = gl + G * j == kr ? eig_one<MODE>() : eig_zero<MODE>();
    u.dim = __ldg(M.blk_dim + u.b);
  } else {
    const int b = __ldcg((half ? C.bblk : C.fblk) + wk.entry);
    u.vanished = b < 0;
    u.b = max(b, 0);
    u.dim = __ldg(M.blk_dim + u.b);
    const V *vec = (const V *)(half ? C.bvec : C.fvec) + (size_t)wk.entry * C.dv;
#pragma unroll
    for (int j = 0; j < R; ++j) {
      const int r = gl + G * j;
      u.x[j] = eig_zero<MODE>();
      if (!u.vanished && r < u.dim) {
        if constexpr (MODE == EIG_PAIR) u.x[j].x = __ldcg(vec + r);
        else u.x[j] = __ldcg(vec + r);
      }
    }
    const double2 l = __ldcg((half ? C.blog : C.flog) + wk.entry);
    L0 = l.x - (l.y == 1.0 ? 0.0 : log(l.y));
  }
  // CACHED: the group's states from operator number s0 of the half on are zero
  auto store_zeros = [&](int s0) {
    for (int s = s0 + gl; s < n; s += G) {
      const int ij = half ? wk.i0 - s : wk.i0 + s;
      const bool out = half ? ij >= wk.hi : ij + 1 <= wk.lo;
      const size_t e = wk.eb + (half ? Kn - ij : ij + 1);
      (half ? (out ? C.bblk : C.sbblk) : (out ? C.fblk : C.sfblk))[e] = -1;
      (half ? (out ? C.blog : C.sblog) : (out ? C.flog : C.sflog))[e] = make_double2(0.0, 1.0);
    }
  };
  if constexpr (CACHED) {
    // A half that starts from a zero state stays zero, and its entry names no block: it follows no
    // operators (block 0 and its key would lead to operators without a target, whose block -1 must
    // never index a table) and stands on block 0 to the end.
    if (u.vanished) {
      if (wk.store) store_zeros(0);
      n = 0;
    }
  }
  if constexpr (CACHED) {
    // the interval from a cached state to the first operator
    const bool act = on && wk.entry >= 0 && !u.vanished;
    EigDt dt{0.f, 0.f, act ? (half ? wk.t0 - tf : tf - wk.t0) : 0.0};
    if (act) L0 = fma(-dt.d, __ldg(M.eig_base + u.b), L0);
    dt.h = (float)dt.d;
    dt.l = (float)(dt.d - (double)dt.h);
    const int eo = __ldg(M.blk_off + u.b);
    E wt[R];
#pragma unroll
    for (int j = 0; j < R; ++j) wt[j] = gl + G * j < u.dim ? eig_weight<MODE>(M, eig_lambda<MODE>(M, eo + gl + G * j), dt) : eig_zero<MODE>();
    if (!eig_interval<MODE, G, R>(M, u.x, wt, act, gl, eo, u.dim, dt, Lx, ex, sc)) u.vanished = true;
  }
  const int key = __ldg(M.blk_key + u.b);
  int nn = key & 0xfffff, mk = key >> 20;
#pragma unroll
  for (int j = 0; j < R; ++j) {
    const int r = gl + G * j;
    if (r < DP) xs[r] = u.x[j];
  }
  __syncwarp();
  const int nmax = G == 32 ? n : __reduce_max_sync(FULL, n);
  int cb = 0;
  bool fock = false;  // the vector is in the occupation basis (operators at equal times)
  // Small blocks (a row per lane, at most 12): the row of the next operator's matrix and its eigenvalue are
  // loaded as soon as the current row is used, and the weights are formed beside the products, so that
  // the chain from one vector to the next holds neither a load nor an exponential. The next G operators'
  // times and flavors are read one turn ahead. 16 steps of 1,024 five-orbital chains 2,660 -> 2,390 us
  // (cached 2,738 -> 2,300), 777 five-orbital ratios 77 -> 61, 4,096 in FP64 457 -> 376 us. It wants 128
  // registers: with a warp per walker four CTAs of four warps per SM, where five at 96 registers (spills)
  // take 429 us for the FP64 ratios and seven without the read-ahead 453.
  constexpr bool PRE = R == 1 && NV <= 6;
  float4 row[PRE ? NV : 1];
  E lam = eig_zero<MODE>();
  if constexpr (PRE)
#pragma unroll
    for (int v = 0; v < NV; ++v) row[v] = make_float4(0.f, 0.f, 0.f, 0.f);
  auto fetch = [&](int mo, int pj) {
    const int ds = (pj >> 16) & 63, dd = (pj >> 22) & 63, nv = (ds + T::EPV - 1) / T::EPV;
    if (gl < dd) {
      const float4 *p = (const float4 *)M.eig_mat + (size_t)mo + gl * nv;
#pragma unroll
      for (int v = 0; v < (PRE ? NV : 1); ++v)
        if (v < nv) row[v] = __ldg(p + v);
      lam = eig_lambda<MODE>(M, (pj & 0xffff) + gl);
    }
  };
  Op op_next{0.0, 0, 0};
  double t_next = 0.0;
  auto fetch_ops = [&](int s) {
    if (s < n) {
      const int idx = half ? wk.i0 - s : wk.i0 + s;
      op_next = cur.get(idx);
      t_next = s + 1 == n ? wk.t_end : cur.get(half ? idx - 1 : idx + 1).t;
    }
  };
  if constexpr (PRE) fetch_ops(gl);
  double Ll = 0.0;  // per lane: its operators' share of the log-weight; CACHED: the group's sum so far
  for (int base = 0; base < nmax; base += G) {
    // the next G operators of the half, one per lane
    const int s = base + gl;
    const bool have = s < n;
    if constexpr (!PRE) fetch_ops(s);
    int moff = 0, pk = 0, tgt = 0, code = 0;
    EigDt dt{0.f, 0.f, 0.0};
    if (have) {
      dt.d = half ? op_next.t - t_next : t_next - op_next.t;
      code = 2 * op_next.f + (half ? 1 - op_next.dag : op_next.dag);
    }
    if constexpr (PRE) fetch_ops(s + G);
    const int dn = have ? key_step(code) : 0, dm = have ? (1 << (code >> 2)) & M.key_mask : 0;
    int pn = dn, pm = dm;
    key_scan<G>(pn, pm, gl);
    double Lop = 0.0;
    if (have) {
      const int b = key_block(M, nn + pn - dn, mk ^ pm ^ dm);
      int4 e = make_int4(0, 0, -1, 0);
      if (!CACHED || b >= 0) e = __ldg(M.eig_op + (size_t)max(b, 0) * 2 * M.nf + code);
      moff = e.x;
      pk = e.y;
      tgt = e.z;
      Lop = -dt.d * __ldg(M.eig_base + max(tgt, 0));
      if (dt.d == 0.0 && s + 1 < n) pk |= 1 << 28;  // at the same time as the next operator
      if constexpr (MODE != EIG_F64) {
        dt.h = (float)dt.d;
        dt.l = (float)(dt.d - (double)dt.h);
      }
    }
    nn += __shfl_sync(FULL, pn, G - 1, G);
    mk ^= __shfl_sync(FULL, pm, G - 1, G);
    int dead = G;  // CACHED: the first of these operators without a target block
    if constexpr (CACHED) {
      const unsigned bad = __ballot_sync(FULL, have && tgt < 0) >> (lane / G * G);
      const unsigned gb = G == 32 ? bad : bad & ((1u << (G & 31)) - 1u);
      if (gb) dead = __ffs(gb) - 1;
    }
    double Lpre = 0.0;  // CACHED: log-weight collected before this lane's operator
    if constexpr (CACHED) {
      double sum = Lop;
#pragma unroll
      for (int o = 1; o < G; o <<= 1) {
        const double a = __shfl_up_sync(FULL, sum, o, G);
        if (gl >= o) sum += a;
      }
      Lpre = Ll + (sum - Lop);
      Ll += __shfl_sync(FULL, sum, G - 1, G);
    } else {
      Ll += Lop;
    }
    const int cnt = min(G, nmax - base);
    int Ej = 0;  // CACHED: the power of two and the shift when this lane's operator was done
    double Lj = 0.0;
    bool vj = false;
    if constexpr (PRE) fetch(__shfl_sync(FULL, moff, 0, G), __shfl_sync(FULL, pk, 0, G));
    for (int j = 0; j < cnt; ++j) {
      if (CACHED && j >= dead) u.vanished = true;
      const bool act = base + j < n && !(CACHED && u.vanished);
      const int mo = __shfl_sync(FULL, moff, j, G), pj = __shfl_sync(FULL, pk, j, G);
      EigDt dj{0.f, 0.f, 0.0};
      if constexpr (MODE == EIG_F64) {
        dj.d = __shfl_sync(FULL, dt.d, j, G);
      } else {
        dj.h = __shfl_sync(FULL, dt.h, j, G);
        dj.l = __shfl_sync(FULL, dt.l, j, G);
      }
      const int eoff = pj & 0xffff, ds = (pj >> 16) & 63, dd = (pj >> 22) & 63;
      const float4 *xv = reinterpret_cast<const float4 *>(xs + cb * DP);
      E acc[R], wt[R];
      if constexpr (PRE) {
        wt[0] = eig_weight<MODE>(M, lam, dj);
        if constexpr (MODE == EIG_PAIR) {
          // vectors past the source's rows meet zeros of xs; the second half is left out where neither
          // group of the warp needs it
          float a[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
          for (int v = 0; v < NV / 2; ++v) eig_fma4(a, row[v], xv[v]);
          if (__any_sync(FULL, ds > NV / 2 * T::EPV))
#pragma unroll
            for (int v = NV / 2; v < NV; ++v) eig_fma4(a, row[v], xv[v]);
          float h, l;
          eig_two_sum(a[0], (a[1] + a[2]) + a[3], h, l);
          acc[0] = make_float2(h, l);
        } else {
          acc[0] = eig_zero<MODE>();
          const int nv = (ds + T::EPV - 1) / T::EPV;
#pragma unroll
          for (int v = 0; v < NV; ++v)
            if (v < nv) eig_fma<MODE>(acc[0], row[v], xv[v]);
        }
        if (gl >= dd) acc[0] = eig_zero<MODE>();
        if (j + 1 < cnt) fetch(__shfl_sync(FULL, moff, j + 1, G), __shfl_sync(FULL, pk, j + 1, G));
      } else {
        const int nv = (ds + T::EPV - 1) / T::EPV;
#pragma unroll
        for (int i = 0; i < R; ++i) {
          acc[i] = eig_zero<MODE>();
          const int r = gl + G * i;
          if (r < dd) {
            const float4 *p = (const float4 *)M.eig_mat + (size_t)mo + r * nv;
            if constexpr (NV <= 6) {
#pragma unroll
              for (int v = 0; v < NV; ++v)
                if (v < nv) eig_fma<MODE>(acc[i], __ldg(p + v), xv[v]);
            } else {
#pragma unroll 6
              for (int v = 0; v < nv; ++v) eig_fma<MODE>(acc[i], __ldg(p + v), xv[v]);
            }
            if constexpr (MODE == EIG_PAIR) {
              float h, l;
              eig_two_sum(acc[i].x, acc[i].y, h, l);
              acc[i] = make_float2(h, l);
            }
          }
        }
      }
      const bool tied = act && (pj >> 28) != 0;
      if (__any_sync(FULL, tied || fock)) {
        const bool here = act && (tied || fock);
        const int tj = __shfl_sync(FULL, tgt, j, G), cj = __shfl_sync(FULL, code, j, G);
        // the source block: the target of the operator before
        const int tp = __shfl_sync(FULL, tgt, max(j - 1, 0), G), bs = j > 0 ? tp : u.b;
        eig_tied<MODE, G, DMAX>(M, xs, cb, here, fock, here ? bs : 0, here ? tj : 0, cj);
        if (here) {
          fock = tied;
#pragma unroll
          for (int i = 0; i < R; ++i) {
            const int r = gl + G * i;
            if (r < DP) {
              acc[i] = xs[(cb ^ 1) * DP + r];
              if (fock) u.x[i] = xs[cb * DP + r];
            }
          }
        }
        __syncwarp();
      }
      if (act && !fock)
#pragma unroll
        for (int i = 0; i < R; ++i) u.x[i] = acc[i];
      if (CACHED && wk.store && base + j < n) {
        // the state right after this operator
        const int ij = half ? wk.i0 - base - j : wk.i0 + base + j;
        const bool out = half ? ij >= wk.hi : ij + 1 <= wk.lo;
        const size_t e = wk.eb + (half ? Kn - ij : ij + 1);
        V *vec = (V *)(half ? (out ? C.bvec : C.sbvec) : (out ? C.fvec : C.sfvec)) + e * C.dv;
        if (!u.vanished)
#pragma unroll
          for (int i = 0; i < R; ++i) {
            const int r = gl + G * i;
            if (r < dd) {
              if constexpr (MODE == EIG_PAIR) vec[r] = acc[i].x + acc[i].y;
              else vec[r] = acc[i];
            }
          }
        if (gl == j) {
          Ej = ex;
          Lj = Lx;
          vj = u.vanished;
        }
      }
      if constexpr (!PRE)
#pragma unroll
        for (int i = 0; i < R; ++i)
          wt[i] = gl + G * i < dd ? eig_weight<MODE>(M, eig_lambda<MODE>(M, eoff + gl + G * i), dj) : eig_zero<MODE>();
      if (!eig_interval<MODE, G, R>(M, u.x, wt, act && !u.vanished && !fock, gl, eoff, dd, dj, Lx, ex, sc)) u.vanished = true;
      cb ^= 1;
#pragma unroll
      for (int i = 0; i < R; ++i) {
        const int r = gl + G * i;
        if (r < DP) xs[cb * DP + r] = u.x[i];
      }
      __syncwarp();
      if (act) u.dim = dd;
    }
    if (CACHED && wk.store && have) {
      // log-weights and blocks of the states stored in this turn, all lanes at once: four FP64
      // instructions for G states, where one lane per operator spent them on every operator
      const int ij = half ? wk.i0 - s : wk.i0 + s;
      const bool out = half ? ij >= wk.hi : ij + 1 <= wk.lo;
      const size_t e = wk.eb + (half ? Kn - ij : ij + 1);
      double2 *lg = half ? (out ? C.blog : C.sblog) : (out ? C.flog : C.sflog);
      int32_t *bk = half ? (out ? C.bblk : C.sbblk) : (out ? C.fblk : C.sfblk);
      bk[e] = vj ? -1 : tgt;
      lg[e] = make_double2(vj ? 0.0 : L0 + Lpre + Lj + (double)Ej * 0.69314718055994530942, 1.0);
    }
    const int last = min(n - base, G) - 1;  // the block after the group's last operator so far
    const int tl = __shfl_sync(FULL, tgt, max(last, 0), G);
    if (last >= 0) u.b = CACHED ? max(tl, 0) : tl;
    if constexpr (BUILD) {
      // every group's path has broken: the states that are left are zero
      if (__all_sync(FULL, u.vanished || base + G >= n)) {
        if (wk.store && u.vanished) store_zeros(base + G);
        break;
      }
    }
  }
  if constexpr (CACHED) {
    if (u.vanished) {  // no block of its own
      u.b = 0;
      u.dim = __ldg(M.blk_dim);
    }
  } else {
#pragma unroll
    for (int o = G / 2; o > 0; o >>= 1) Ll += __shfl_xor_sync(FULL, Ll, o);
  }
  u.L = L0 + Ll + Lx + (double)ex * 0.69314718055994530942;
}

// Rows of a vector in the occupation basis: (V x)_r = sum_k V_k[r] x_k, from the components x in
// shared memory (double, `dim` of them).
__device__ __forceinline__ double eig_fock_row(const DevModel &M, int b, int dim, int r, const double *x) {
  const double *V = M.blk_evec64 + __ldg(M.blk_evoff + b);
  double a = 0.0;
  for (int k = 0; k < dim; ++k) a = fma(__ldg(V + k * dim + r), x[k], a);
  return a;
}

// ---------------------------------------------------------------------------
// The whole call of a walker: validation, edit, structural pruning, items, reduction
// ---------------------------------------------------------------------------
// SOLO: one warp per walker, several walkers per CTA. Otherwise one CTA per walker: every warp
// repeats the validation and the pruning (integer work on data in L1) and takes every
// NW-th of the surviving items, so that no list, counter or second launch is needed.
// G lanes serve one half of an item; with G <= 16 both halves of an item sit in one warp and
// run in step, with G = 32 in two neighbouring warps that meet at a named barrier.
template <int MODE, int G, int DMAX, bool SOLO>
struct EigShared {
  static constexpr int DP = EigHalf<MODE, G, DMAX>::DP;
  static constexpr int GW = 32 / G;                  // groups per warp
  static constexpr int IPW = G == 32 ? 1 : GW / 2;   // items per warp (G = 32: per pair of warps)
  static constexpr int WPI = G == 32 ? 2 : 1;        // warps per item
  static constexpr int NWM = SOLO ? 4 : 8;           // warps per CTA at most
  typename EigT<MODE>::E xs[NWM * GW * 2 * DP];
  double pd[NWM * GW * DP];                          // final vectors (G = 32, observables)
  double res_log[64 * (SOLO ? NWM : 1)];
  int res_sgn[64 * (SOLO ? NWM : 1)];
  double half_log[NWM];
};

// The two warps of an item (G = 32) or the lanes of a warp meet.
template <int G>
__device__ __forceinline__ void eig_meet() {
  if constexpr (G == 32) asm volatile("bar.sync %0, 64;" ::"r"(1 + (int)(threadIdx.x >> 6)) : "memory");
  else __syncwarp();
}

// Structural pruning of up to 64 kept states from q0 on: the lanes take one operator each, and a
// kept state survives while the key after every operator has a block. Bit q: q0 + q survives.
__device__ __forceinline__ unsigned long long eig_alive(const DevModel &M, const Cursor &cur, int Kn, int q0, int nq,
                                                        int lane) {
  unsigned long long alive = nq == 64 ? ~0ull : (1ull << nq) - 1;
  int nn = 0, mk = 0;
  for (int base = 0; base < Kn && alive; base += 32) {
    const bool have = base + lane < Kn;
    int code = 0;
    if (have) {
      const Op op = cur.get(base + lane);
      code = 2 * op.f + op.dag;
    }
    int pn = have ? key_step(code) : 0, pm = have ? (1 << (code >> 2)) & M.key_mask : 0;
    key_scan<32>(pn, pm, lane);
    pn += nn;
    pm ^= mk;
    for (unsigned long long todo = alive; todo; todo &= todo - 1) {
      const int q = __ffsll((long long)todo) - 1;
      const int k0 = __ldg(M.kept_key + q0 + q);
      const bool bad = have && key_block(M, (k0 & 0xfffff) + pn, (k0 >> 20) ^ pm) < 0;
      if (__any_sync(FULL, bad)) alive &= ~(1ull << q);
    }
    nn = __shfl_sync(FULL, pn, 31);
    mk = __shfl_sync(FULL, pm, 31);
  }
  return nn != 0 || mk != 0 ? 0ull : alive;
}

// Overlap of the two halves of an item, its log-weight and sign (all lanes of half 0 hold them).
// MEAS: into the workspace the matrix elements of the observables between the halves, their
// overlap (half_log) and their common log-weight (item_log). The elements are not divided by the overlap:
// a singlet and a triplet have none, but n_f and S_z have elements between them.
template <int MODE, int G, int DMAX, bool MEAS, typename SH>
__device__ __forceinline__ void eig_overlap(const DevModel &M, const Workspace &ws, SH &sh, EigHalf<MODE, G, DMAX> &u,
                                            bool on, int half, int item, double &L, int &sgn) {
  using H = EigHalf<MODE, G, DMAX>;
  constexpr int DP = H::DP, R = H::R;
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5, grp = lane / G, gl = lane % G;
  double ov = 0.0, Lo;
  bool van;
  if constexpr (G == 32) {
    double *mine = sh.pd + (size_t)wib * DP;
#pragma unroll
    for (int j = 0; j < R; ++j) {
      const int r = gl + G * j;
      if (r < DP) mine[r] = eig_value<MODE>(u.x[j]);
    }
    if (lane == 0) sh.half_log[wib] = u.vanished ? -INFINITY : u.L;
    eig_meet<G>();
    const double *oth = sh.pd + (size_t)(wib ^ 1) * DP;
    Lo = sh.half_log[wib ^ 1];
    van = u.vanished || Lo == -INFINITY;
#pragma unroll
    for (int j = 0; j < R; ++j) {
      const int r = gl + G * j;
      if (r < u.dim) ov = fma(eig_value<MODE>(u.x[j]), oth[r], ov);
    }
  } else {
    Lo = __shfl_xor_sync(FULL, u.L, G);
    const bool vo = __shfl_xor_sync(FULL, (int)u.vanished, G) != 0;
    van = u.vanished || vo;
#pragma unroll
    for (int j = 0; j < R; ++j) {
      const double a = eig_value<MODE>(u.x[j]);
      ov = fma(a, __shfl_xor_sync(FULL, a, G), ov);
    }
  }
#pragma unroll
  for (int o = G / 2; o > 0; o >>= 1) ov += __shfl_xor_sync(FULL, ov, o);
  const bool zero = van || ov == 0.0;
  L = zero ? -INFINITY : u.L + Lo + log(fabs(ov));
  sgn = zero ? 0 : (ov > 0.0 ? 1 : -1);
  if constexpr (MEAS) {
    // the halves in the occupation basis: each replaces its own components
    double *own = sh.pd + (size_t)(G == 32 ? wib : wib * (32 / G) + grp) * DP;
    const double *fv = sh.pd + (size_t)(G == 32 ? wib & ~1 : wib * (32 / G) + (grp & ~1)) * DP, *bv = fv + DP;
    if constexpr (G != 32) {
#pragma unroll
      for (int j = 0; j < R; ++j) {
        const int r = gl + G * j;
        if (r < DP) own[r] = eig_value<MODE>(u.x[j]);
      }
      __syncwarp();
    }
    double fr[R];
#pragma unroll
    for (int j = 0; j < R; ++j) {
      const int r = gl + G * j;
      fr[j] = on && r < u.dim ? eig_fock_row(M, u.b, u.dim, r, own) : 0.0;
    }
    eig_meet<G>();
#pragma unroll
    for (int j = 0; j < R; ++j) {
      const int r = gl + G * j;
      if (r < DP) own[r] = fr[j];
    }
    eig_meet<G>();
    if (on && half == 0) {
      // n_f and double occupancies, one lane each
      const int nl = M.nf + M.n_orb + 1, off = __ldg(M.blk_off + u.b);
      double *io = ws.item_obs + (size_t)item * nl;
      for (int k = gl; k < nl - 1; k += G) {
        const int bit = k < M.nf ? k : 2 * (k - M.nf), msk = k < M.nf ? 1 : 3;
        double a = 0.0;
        for (int r = 0; r < u.dim; ++r)
          if (((__ldg(M.st_bits + off + r) >> bit) & msk) == msk) a = fma(fv[r], bv[r], a);
        io[k] = a;
      }
      // S^2: sum_r backward_r (S^2 forward)_r
      const int s2w = __ldg(M.blk_s2w + u.b), s2o = __ldg(M.blk_s2ell + u.b);
      double a = 0.0;
      for (int r = gl; r < u.dim; r += G) {
        double t = (double)__ldg(M.s2_diag + off + r) * fv[r];
        for (int k = 0; k < s2w; ++k) {
          const unsigned e = __ldg(M.s2_ell + s2o + k * u.dim + r);
          if (e != 0xFFFFu) t += (e & 0x8000u) ? -fv[e & 0x7fffu] : fv[e & 0x7fffu];
        }
        a = fma(t, bv[r], a);
      }
      const unsigned hm = G == 32 ? FULL : (((1u << (G & 31)) - 1u) << (grp * G));
#pragma unroll
      for (int o = G / 2; o > 0; o >>= 1) a += __shfl_xor_sync(hm, a, o);
      if (gl == 0) {
        io[nl - 1] = a;
        ws.item_blk[item] = u.b;
        ws.item_log[item] = van ? -INFINITY : u.L + Lo;
        ws.half_log[item] = ov;
        ws.item_sign[item] = van ? 0 : 1;  // whether the item takes part
      }
    }
  }
  if constexpr (G == 32 || MEAS) eig_meet<G>();
}

// Signed log-sum-exp of up to 64 items' (log, sign) into (mx, acc), in the order of the kept
// states, by one warp.
__device__ __forceinline__ void eig_accumulate(const double *rl, const int *rs, int na, int lane, double &mx,
                                               double &acc, int &wst) {
  double bm = mx;
  for (int i = lane; i < na; i += 32)
    if (rs[i] != 0) {
      if (!isfinite(rl[i])) wst = KT_ENUMERIC;
      bm = fmax(bm, rl[i]);
    }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) bm = fmax(bm, __shfl_xor_sync(FULL, bm, o));
  if (!(bm > -INFINITY)) return;
  if (na == 1 && mx == -INFINITY) {
    acc = (double)rs[0];
  } else {
    double a = 0.0;
    for (int i = lane; i < na; i += 32)
      if (rs[i] != 0) a += (double)rs[i] * exp(rl[i] - bm);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) a += __shfl_xor_sync(FULL, a, o);
    acc = (mx > -INFINITY ? acc * exp(mx - bm) : 0.0) + a;
  }
  mx = bm;
}

// A walker's outputs from the sum over its items.
__device__ __forceinline__ void eig_output(const DevModel &M, int w, int has_moves, const int8_t *cur_sign,
                                           const double *cur_logabs, double mx, double acc, int wst, int8_t *sign,
                                           double *logv, int32_t *status) {
  int sg = 0;
  double la = -INFINITY;
  if (acc != 0.0 && isfinite(mx)) {
    sg = acc > 0.0 ? 1 : -1;
    la = mx + (fabs(acc) == 1.0 ? 0.0 : log(fabs(acc))) - M.beta * M.E0;
  }
  if (has_moves) {
    sign[w] = (int8_t)(sg * cur_sign[w]);
    logv[w] = sg != 0 ? la - cur_logabs[w] : -INFINITY;
  } else {
    sign[w] = (int8_t)sg;
    logv[w] = la;
  }
  if (sg != 0 && !isfinite(la)) wst = KT_ENUMERIC;
  status[w] = wst;
}

// What to do with the cache: nothing, ratios from it (read only, or keeping this step's states),
// store every state of the current configurations, or the observables at beta/2.
constexpr int EIG_PLAIN = 0, EIG_RATIO = 1, EIG_BUILD = 2, EIG_MEASURE = 3;

template <int MODE, int G, int DMAX, bool MEAS, int CACHE, bool SOLO>
__global__ void __launch_bounds__(SOLO ? 128 : 256, SOLO ? 4 : 2)
    eig_kernel(DevModel M, SeqView S, MoveView mv, int has_moves, const int8_t *cur_sign, const double *cur_logabs,
               Workspace ws, CacheView C, int write, int8_t *sign, double *logv, int32_t *status, double *obs) {
  using H = EigHalf<MODE, G, DMAX>;
  using SH = EigShared<MODE, G, DMAX, SOLO>;
  constexpr int DP = H::DP, GW = SH::GW, IPW = SH::IPW, WPI = SH::WPI;
  constexpr bool BUILD = CACHE == EIG_BUILD;
  static_assert(!(SOLO && G == 32), "an item of two warps needs a CTA");
  __shared__ __align__(16) SH sh;
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const int grp = lane / G, gl = lane % G;
  const int half = G == 32 ? wib & 1 : grp & 1;
  const int w = SOLO ? (int)(blockIdx.x * nw + wib) : (int)blockIdx.x;
  if (SOLO && w >= S.n) return;
  const int nk = M.n_kept, nl = M.nf + M.n_orb + 1;
  const int tid = SOLO ? lane : (int)threadIdx.x, nt = SOLO ? 32 : (int)blockDim.x;
  int4 d;
  const int st = prep_walker(M, S, mv, has_moves, cur_sign, w, lane, d);
  if (tid == 0) {
    ws.desc[w] = d;
    ws.wstatus[w] = st;
  }
  const int nobs = MEAS ? nl + (M.n_orb + 1) * (M.n_orb + 1) : 0;
  if (st != KT_OK) {
    if (!BUILD && tid == 0) {
      sign[w] = 0;
      logv[w] = (st == KT_EZEROWEIGHT || st == KT_EINVAL) ? NAN : -INFINITY;
      status[w] = st;
    }
    if (MEAS)
      for (int k = tid; k < nobs; k += nt) obs[(size_t)w * nobs + k] = NAN;
    if (BUILD)
      for (int q = tid; q < nk; q += nt) C.f[w * nk + q] = C.gr[w * nk + q] = 0;
    return;
  }
  Cursor cur;
  cur.S = S;
  cur.o = __ldg(S.offsets + w);
  cur.d = d;
  set_cursor_move(cur, mv, has_moves != 0, w);
  const int Kn = d.w;
  // where the halves meet: the middle operator of the stretch, or beta/2 for the observables
  int m = 0;
  double t_s = 0.0;
  if (MEAS) {
    t_s = 0.5 * M.beta;
    for (int base = 0; base < Kn; base += 32) {
      const int i = base + lane;
      m += __popc(__ballot_sync(FULL, i < Kn && __ldg(S.tau + cur.o + i) < t_s));
    }
  } else if (CACHE == EIG_PLAIN) {
    m = Kn / 2 > 1 ? Kn / 2 : (Kn > 0 ? 1 : 0);
    t_s = Kn > 0 ? cur.get(m - 1).t : 0.0;
    while (m < Kn && cur.get(m).t == t_s) ++m;  // operators at equal times stay in one half
  }
  // the cache: the edited window, and whether this walker uses it
  const int Ko = !has_moves ? Kn : (d.x == 0 ? Kn - 2 : Kn + 2);
  int lo = Kn, hi = 0;
  if (CACHE == EIG_RATIO) edit_window(d, lo, hi);
  const bool fits = CACHE != EIG_PLAIN && Kn <= C.P && Ko <= C.P;
  if (BUILD) {
    for (int q = tid; q < nk; q += nt) C.f[w * nk + q] = C.gr[w * nk + q] = fits ? Kn : 0;
    if (!fits) return;
  }
  typename EigT<MODE>::E *xs = sh.xs + (size_t)(wib * GW + grp) * 2 * DP;
  double *rl = sh.res_log + (SOLO ? 64 * wib : 0);
  int *rs = sh.res_sgn + (SOLO ? 64 * wib : 0);
  double mx = -INFINITY, acc = 0.0;
  int wst = KT_OK;
  for (int q0 = 0; q0 < nk; q0 += 64) {
    const int nq = min(64, nk - q0);
    const unsigned long long alive =
        BUILD ? (nq == 64 ? ~0ull : (1ull << nq) - 1) : eig_alive(M, cur, Kn, q0, nq, lane);
    if (MEAS) {
      // the pruned items count as zero; a surviving item's sign is written by its own warp only (nothing
      // orders the warps before the reduction)
      for (int q = tid; q < nq; q += nt)
        if (!((alive >> q) & 1)) ws.item_sign[(size_t)w * nk + q0 + q] = 0;
    }
    if (CACHE == EIG_RATIO && write) {
      // the commit of an accepted move needs the plan of the items that are zero now, too
      for (int q = tid; q < nq; q += nt)
        if (!((alive >> q) & 1)) C.plan[(size_t)w * nk + q0 + q] = make_int4(0, 0, 0, fits ? 1 : 0);
    }
    const int na = __popcll(alive);
    // items, `step` at a time
    const int step = SOLO ? IPW : (nw / WPI) * IPW;
    for (int r0 = 0; r0 < na; r0 += step) {
      const int rank = r0 + (SOLO ? 0 : (wib / WPI) * IPW) + (G == 32 ? 0 : grp >> 1);
      const bool on = rank < na;
      unsigned long long t = alive;
      for (int i = 0; i < (on ? rank : 0); ++i) t &= t - 1;
      const int q = q0 + (on ? __ffsll((long long)t) - 1 : 0);
      const int item = w * nk + q;
      EigWork wk;
      wk.half = half;
      wk.q = q;
      wk.entry = -1;
      wk.t_end = t_s;
      wk.store = false;
      bool cached = false;
      if constexpr (CACHE == EIG_PLAIN) {
        wk.i0 = half ? Kn - 1 : 0;
        wk.n = on ? (half ? Kn - m : m) : -1;
      } else {
        // the stretch [y, x) of operators between a valid forward and a valid backward state
        int y = 0, x = Kn;
        cached = on && fits;
        if (cached && !BUILD) {
          const int f = __ldcg(C.f + item), gr = __ldcg(C.gr + item);
          // read-only use (fixed configurations): the cache was built for every operator of the
          // current sequence, so a walker whose length differs from the build is evaluated in full
          if (CACHE == EIG_RATIO && !write && f != Ko) cached = false;
          if (cached) {
            y = min(MEAS ? m : lo, f);
            x = MEAS ? max(m, Kn - gr) : max(hi - (Kn - Ko), Ko - gr) + (Kn - Ko);
            // operators at equal times are taken together
            while (y > 0 && y < Kn && cur.get(y - 1).t == cur.get(y).t) --y;
            while (x > 0 && x < Kn && cur.get(x - 1).t == cur.get(x).t) ++x;
          }
        }
        int me = m;
        if (CACHE == EIG_RATIO) {
          me = y + (x - y) / 2;
          while (me > 0 && me < x && cur.get(me - 1).t == cur.get(me).t) ++me;
          if (write && on && half == 0 && gl == 0) C.plan[item] = make_int4(y, x, me, (cached ? 1 : 0) | 2);
          wk.t_end = me >= 1 ? cur.get(me - 1).t : 0.0;
        }
        wk.i0 = half ? x - 1 : y;
        wk.n = on ? (BUILD ? Kn : (half ? x - me : me - y)) : -1;
        if (BUILD) wk.t_end = Kn > 0 ? cur.get(half ? 0 : Kn - 1).t : 0.0;
        wk.eb = (size_t)item * ((size_t)C.P + 1);
        wk.lo = lo;
        wk.hi = hi;
        wk.store = cached && (CACHE != EIG_RATIO || write);
        if (on && (half ? x < Kn : y > 0)) {
          wk.entry = (long long)(wk.eb + (half ? Kn - x : y));
          wk.t0 = cur.get(half ? x : y - 1).t;
        }
      }
      H u;
      eig_half<MODE, G, DMAX, CACHE != EIG_PLAIN, BUILD>(M, cur, Kn, wk, C, xs, u);
      if constexpr (!BUILD) {
        double L;
        int sg;
        eig_overlap<MODE, G, DMAX, MEAS>(M, ws, sh, u, on, half, item, L, sg);
        if (on && half == 0 && gl == 0) {
          rl[rank] = L;
          rs[rank] = sg;
        }
        if (CACHE == EIG_MEASURE && cached && gl == 0) {
          // the states passed belong to the current configuration: the valid range grows
          if (half == 0) C.f[item] = max(C.f[item], m);
          else C.gr[item] = max(C.gr[item], Kn - m);
        }
      }
    }
    if constexpr (!BUILD) {
      if (SOLO) __syncwarp();
      else __syncthreads();
      if (SOLO || wib == 0) eig_accumulate(rl, rs, na, lane, mx, acc, wst);
      if (SOLO) __syncwarp();
      else __syncthreads();
    }
  }
  if (BUILD || !(SOLO || wib == 0)) return;
  wst = __reduce_max_sync(FULL, wst);
  if (lane == 0) eig_output(M, w, has_moves, cur_sign, cur_logabs, mx, acc, wst, sign, logv, status);
  if constexpr (MEAS) {
    // sums over the items of weight times element, in units of exp(mx), over the trace in the same units;
    // the (n_up, n_dn) histogram adds the overlaps
    double *out = obs + (size_t)w * nobs;
    const bool some = acc != 0.0 && isfinite(mx);
    for (int k = lane; k < nobs; k += 32) {
      double a = 0.0, den = 0.0;
      for (int q = 0; q < nk; ++q) {
        const int item = w * nk + q;
        if (ws.item_sign[item] == 0) continue;
        const double c = exp(ws.item_log[item] - mx), ov = ws.half_log[item];
        double e = 0.0;
        if (k < nl) {
          e = ws.item_obs[(size_t)item * nl + k];
        } else {
          const int x = __ldg(M.st_bits + __ldg(M.blk_off + ws.item_blk[item]));
          if (__popc(x & 0x5555) * (M.n_orb + 1) + __popc(x & 0xaaaa) == k - nl) e = ov;
        }
        if (e != 0.0) a = fma(c, e, a);    // c may be huge where both elements are zero
        if (ov != 0.0) den = fma(c, ov, den);
      }
      out[k] = some ? a / (den != 0.0 ? den : acc) : NAN;
    }
  }
}

// Arguments of one launch (what each call leaves out stays null).
struct EigCall {
  SeqView S;
  MoveView mv;
  int has_moves;
  const int8_t *cur_sign;
  const double *cur_logabs;
  Workspace ws;
  CacheView C;
  int write;
  int8_t *sign;
  double *logv;
  int32_t *status;
  double *obs;
};

// Launch shape. A batch that fills the chip with a warp per walker takes four walkers per CTA.
// Smaller batches, and items of two warps, take one CTA per walker, with as many warps as
// bring about 16 per SM or as there are kept states to share out.
template <int MODE, int G, int DMAX, bool MEAS, int CACHE>
int launch_eig(const DevModel &M, const EigCall &c, cudaStream_t st) {
  constexpr int IPW = G == 32 ? 1 : 16 / G, WPI = G == 32 ? 2 : 1;
  const int share = std::min((M.n_kept + IPW - 1) / IPW, 152 * 16 / WPI / std::max(c.S.n, 1));
  const int want = std::min(8 / WPI, std::max(1, share)) * WPI;
  if constexpr (G != 32) {
    if (want == 1) {
      eig_kernel<MODE, G, DMAX, MEAS, CACHE, true><<<(unsigned)((c.S.n + 3) / 4), 128, 0, st>>>(
          M, c.S, c.mv, c.has_moves, c.cur_sign, c.cur_logabs, c.ws, c.C, c.write, c.sign, c.logv, c.status, c.obs);
      return (int)cudaGetLastError();
    }
  }
  eig_kernel<MODE, G, DMAX, MEAS, CACHE, false><<<(unsigned)c.S.n, want * 32, 0, st>>>(
      M, c.S, c.mv, c.has_moves, c.cur_sign, c.cur_logabs, c.ws, c.C, c.write, c.sign, c.logv, c.status, c.obs);
  return (int)cudaGetLastError();
}

}  // namespace dev
}  // namespace kt
