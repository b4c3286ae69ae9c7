// Operator matrices between the block eigenbases, and the dispatch of the calls that use them.
#include "kt_eig.cuh"

namespace kt {

int dispatch_eig_f32(int kd, int G, int cache, const DevModel &M, const dev::EigCall &c, cudaStream_t st);
int dispatch_eig_f64(int kd, int G, int cache, const DevModel &M, const dev::EigCall &c, cudaStream_t st);

namespace {
using namespace dev;

// Entry (r, k) of the matrix of c_f (dag 0) or c_f^+ (dag 1) from block b to its target: the sum
// over the target's rows i with bit f equal to dag of V_t[i, r] (+-1) V_b[partner(i), k], with vectors
// and sum of two FP64 words each (kt_refine.h). An element that a symmetry of the model forbids
// ends below the bound of its operator (eig_op.w, 1e-25 for the five-orbital model) and is stored as zero: a
// component that a symmetry forbids then stays exactly zero, where the propagator would amplify
// its rounding by exp(dt gap). Elements above it, however small, are the model's (weak hopping, weak
// splitting) and are kept to the accuracy of their format.
template <int MODE>
__global__ void eig_matrix_kernel(DevModel M, const double *__restrict__ evec_lo, typename EigT<MODE>::E *__restrict__ out) {
  constexpr int EPV = EigT<MODE>::EPV;
  const int id = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5), lane = threadIdx.x & 31;
  if (id >= M.n_blocks * M.nf * 2) return;
  const int4 e = M.eig_op[id];
  if (e.z < 0) return;
  const int b = id / (2 * M.nf), f = (id >> 1) % M.nf, dag = id & 1;
  const int d1 = M.blk_dim[b], d2 = M.blk_dim[e.z], off = M.blk_off[e.z];
  const int o1 = M.blk_evoff[b], o2 = M.blk_evoff[e.z];
  const double cut = (double)__int_as_float(e.w);
  const int ld = (d1 + EPV - 1) / EPV * EPV;
  typename EigT<MODE>::E *o = out + (size_t)e.x * EPV;
  for (int i = lane; i < d2 * ld; i += 32) {
    const int r = i / ld, k = i - r * ld;
    double a = 0.0, al = 0.0;
    if (k < d1)
      for (int s = 0; s < d2; ++s)
        if (((M.st_bits[off + s] >> f) & 1) == dag) {
          const unsigned pe = M.partner[(size_t)(off + s) * M.nf + f];
          const int i2 = o2 + r * d2 + s, i1 = o1 + k * d1 + (int)(pe & 0x7fffu);
          const double y = M.blk_evec64[i2], x = (pe & 0x8000u) ? -M.blk_evec64[i1] : M.blk_evec64[i1];
          const double xl = (pe & 0x8000u) ? -evec_lo[i1] : evec_lo[i1];
          const double p = __dmul_rn(y, x);
          const double pl = fma(y, x, -p) + (y * xl + evec_lo[i2] * x);
          // (a, al) += (p, pl)
          const double t = a + p, bb = t - a;
          const double te = (a - (t - bb)) + (p - bb);
          const double u = al + pl, ub = u - al;
          const double ue = (al - (u - ub)) + (pl - ub);
          const double v = te + u, h = t + v, hl = (v - (h - t)) + ue;
          a = h + hl;
          al = hl - (a - h);
        }
    if (fabs(a) < cut) a = 0.0;
    if constexpr (MODE == EIG_PAIR) {
      const double h = rint(a * 2048.0) * (1.0 / 2048.0);
      o[i] = make_float2((float)h, (float)(a - h));
    } else {
      o[i] = (typename EigT<MODE>::E)a;
    }
  }
}

}  // namespace

int build_eig_matrices(const DevModel &M, const double *evec_lo) {
  const unsigned grid = (unsigned)((M.n_blocks * M.nf * 2 + 7) / 8);
  void *o = const_cast<void *>(M.eig_mat);
  switch (M.eig) {
    case EIG_PAIR: eig_matrix_kernel<EIG_PAIR><<<grid, 256>>>(M, evec_lo, (float2 *)o); break;
    case EIG_F64: eig_matrix_kernel<EIG_F64><<<grid, 256>>>(M, evec_lo, (double *)o); break;
  }
  return (int)cudaGetLastError();
}

static int dispatch_eig(int kd, int G, int cache, const DevModel &M, const dev::EigCall &c, void *stream) {
  cudaStream_t st = (cudaStream_t)stream;
  switch (M.eig) {
    case EIG_PAIR: return dispatch_eig_f32(kd, G, cache, M, c, st);
    case EIG_F64: return dispatch_eig_f64(kd, G, cache, M, c, st);
  }
  return (int)cudaErrorInvalidValue;
}

int launch_eig_pipeline(const DevModel &M, int kd, int G, const SeqView &S, const MoveView *moves,
                        const int8_t *cur_sign, const double *cur_logabs, int8_t *sign, double *logv, int32_t *status,
                        const Workspace &ws, void *stream, double *obs) {
  const EigCall c{S, moves ? *moves : MoveView{}, moves ? 1 : 0, cur_sign, cur_logabs, ws, CacheView{}, 0,
                  sign, logv, status, obs};
  return dispatch_eig(kd, G, EIG_PLAIN, M, c, stream);
}

int launch_eig_cached(const DevModel &M, int kd, const SeqView &S, const MoveView &mv, const int8_t *cur_sign,
                      const double *cur_logabs, int8_t *sign, double *logv, int32_t *status, const Workspace &ws,
                      const CacheView &cache, bool write, void *stream) {
  const EigCall c{S, mv, 1, cur_sign, cur_logabs, ws, cache, write ? 1 : 0, sign, logv, status, nullptr};
  return dispatch_eig(kd, 0, EIG_RATIO, M, c, stream);
}

int launch_eig_build(const DevModel &M, int kd, const SeqView &S, const Workspace &ws, const CacheView &cache,
                     void *stream) {
  const EigCall c{S, MoveView{}, 0, nullptr, nullptr, ws, cache, 1, nullptr, nullptr, nullptr, nullptr};
  return dispatch_eig(kd, 0, EIG_BUILD, M, c, stream);
}

int launch_eig_measure(const DevModel &M, int kd, const SeqView &S, int8_t *sign, double *logv, int32_t *status,
                       double *obs, const Workspace &ws, const CacheView &cache, void *stream) {
  const EigCall c{S, MoveView{}, 0, nullptr, nullptr, ws, cache, 1, sign, logv, status, obs};
  return dispatch_eig(kd, 0, EIG_MEASURE, M, c, stream);
}

}  // namespace kt
