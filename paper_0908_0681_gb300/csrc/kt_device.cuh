// Device helpers shared by the kernels of the engine (internal).
#pragma once

#include <cuda_runtime.h>

#include <math.h>
#include <stdint.h>

#include "kt_internal.h"

namespace kt {
namespace dev {


constexpr unsigned FULL = 0xffffffffu;

struct Op {
  double t;
  int f, dag;
};

__device__ __forceinline__ Op load_op(const SeqView &S, int i) {
  return Op{__ldg(S.tau + i), (int)__ldg(S.flavor + i), (int)__ldg(S.dagger + i)};
}

// Operator i of the (possibly edited) sequence of one walker.
// desc = {kind, p1, p2, K_new}: kind -1 none, 0 insert (op A at new index p1,
// op B at new index p2 + 1), 1 remove (old indices p1 < p2 dropped).
struct Cursor {
  SeqView S;
  int o;
  int4 d;
  Op A, B;
  __device__ __forceinline__ Op get(int i) const {
    if (d.x == 0) {
      if (i < d.y) return load_op(S, o + i);
      if (i == d.y) return A;
      if (i <= d.z) return load_op(S, o + i - 1);
      if (i == d.z + 1) return B;
      return load_op(S, o + i - 2);
    }
    if (d.x == 1) {
      if (i < d.y) return load_op(S, o + i);
      if (i < d.z - 1) return load_op(S, o + i + 1);
      return load_op(S, o + i + 2);
    }
    return load_op(S, o + i);
  }
};

// The two operators of walker w's insertion (d.x == 0).
__device__ __forceinline__ void set_cursor_move(Cursor &c, const MoveView &mv, bool has_moves, int w) {
  if (has_moves && c.d.x == 0) {
    const int f = mv.flavor[w];
    const double td = mv.t_dag[w], ta = mv.t_ann[w];
    if (td < ta) {
      c.A = Op{td, f, 1};
      c.B = Op{ta, f, 0};
    } else {
      c.A = Op{ta, f, 0};
      c.B = Op{td, f, 1};
    }
  }
}

__device__ __forceinline__ Cursor make_cursor(const SeqView &S, const MoveView &mv, bool has_moves, const int4 *desc,
                                              int w) {
  Cursor c;
  c.S = S;
  c.o = __ldg(S.offsets + w);
  c.d = desc[w];
  set_cursor_move(c, mv, has_moves, w);
  return c;
}

__device__ __forceinline__ int upper_bound(const double *t, int K, double x) {
  int lo = 0, hi = K;
  while (lo < hi) {
    const int mid = (lo + hi) >> 1;
    if (t[mid] <= x) lo = mid + 1; else hi = mid;
  }
  return lo;
}

// Number of entries of the sorted t[0 .. K) that are < x.
__device__ __forceinline__ int lower_bound(const double *t, int K, double x) {
  int lo = 0, hi = K;
  while (lo < hi) {
    const int mid = (lo + hi) >> 1;
    if (t[mid] < x) lo = mid + 1; else hi = mid;
  }
  return lo;
}

// Validation of walker w's sequence and the edit descriptor of its move, by one warp: the lanes
// read consecutive operators (coalesced) and decide by ballot. Returns the walker's status
// (warp-uniform) and the descriptor (Cursor).
__device__ __forceinline__ int prep_walker(const DevModel &M, const SeqView &S, const MoveView &mv, int has_moves,
                                           const int8_t *cur_sign, int w, int lane, int4 &d) {
  const int o = S.offsets[w], K = S.lens ? S.lens[w] : S.offsets[w + 1] - o;
  int st = KT_OK;
  d = make_int4(-1, 0, 0, K);
  if (K < 0) {
    st = KT_EINVAL;
  } else if (!S.trusted) {
    // times non-decreasing from 0 and below beta, flavors and daggers in range
    double carry = 0.0;
    for (int base = 0; base < K; base += 32) {
      const int i = base + lane;
      double t = 0.0;
      int f = 0, g = 0;
      if (i < K) {
        t = __ldg(S.tau + o + i);
        f = __ldg(S.flavor + o + i);
        g = __ldg(S.dagger + o + i);
      }
      double prev = __shfl_up_sync(FULL, t, 1);
      if (lane == 0) prev = carry;
      const bool bad = i < K && (!(t >= prev) || !(t < M.beta) || f >= M.nf || g > 1);
      if (__any_sync(FULL, bad)) {
        st = KT_EINVAL;
        break;
      }
      carry = __shfl_sync(FULL, t, 31);
    }
  }
  if (has_moves && st == KT_OK) {
    const int kind = mv.kind[w], f = mv.flavor[w];
    if (f >= M.nf) {
      st = KT_EINVAL;
    } else if (kind == 0) {
      const double td = mv.t_dag[w], ta = mv.t_ann[w];
      if (!(td >= 0.0 && td < M.beta && ta >= 0.0 && ta < M.beta)) {
        st = KT_EINVAL;
      } else {
        // insertion points: the number of operators at or before each new time (the sorted
        // sequence's upper bound)
        const double tA = td < ta ? td : ta, tB = td < ta ? ta : td;
        int pa = 0, pb = 0;
        for (int base = 0; base < K; base += 32) {
          const int i = base + lane;
          const double t = i < K ? __ldg(S.tau + o + i) : 0.0;
          pa += __popc(__ballot_sync(FULL, i < K && t <= tA));
          pb += __popc(__ballot_sync(FULL, i < K && t <= tB));
        }
        d = make_int4(0, pa, pb, K + 2);
      }
    } else if (kind == 1) {
      const int r = mv.rem_idx[w];
      if (r < 0 || r >= K || S.flavor[o + r] != f) {
        st = KT_EINVAL;
      } else {
        // its partner: the next operator of the flavor after r, cyclically
        int j = -1;
        for (int base = r + 1; base < K && j < 0; base += 32) {
          const int i = base + lane;
          const unsigned m = __ballot_sync(FULL, i < K && __ldg(S.flavor + o + i) == f);
          if (m) j = base + __ffs(m) - 1;
        }
        for (int base = 0; base < r && j < 0; base += 32) {
          const int i = base + lane;
          const unsigned m = __ballot_sync(FULL, i < r && __ldg(S.flavor + o + i) == f);
          if (m) j = base + __ffs(m) - 1;
        }
        if (j < 0 || S.dagger[o + j] == S.dagger[o + r]) {
          st = KT_EINVAL;
        } else {
          d = make_int4(1, r < j ? r : j, r < j ? j : r, K - 2);
        }
      }
    } else {
      st = KT_EINVAL;
    }
    if (st == KT_OK && cur_sign[w] == 0) st = KT_EZEROWEIGHT;
  }
  return st;
}

__device__ __forceinline__ void stat_add(unsigned long long *p, unsigned long long v) {
  if (v) atomicAdd(p, v);
}

}  // namespace dev
}  // namespace kt
