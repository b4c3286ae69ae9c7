// Traces in the block eigenbasis, EIG_PAIR instances (see kt_eig.cuh): every lane-group size of
// each row capacity for traces and ratios, the default one for observables and the cache.
#include "kt_eig.cuh"

namespace kt {

int dispatch_eig_f32(int kd, int G, int cache, const DevModel &M, const dev::EigCall &c, cudaStream_t st) {
  using namespace dev;
  const bool meas = c.obs != nullptr;
#define KT_EIG_CASE(GG, D, CACHE, MEAS) \
  if (kd == D && cache == CACHE && meas == MEAS && (G == GG || CACHE != EIG_PLAIN || MEAS)) \
    return launch_eig<EIG_PAIR, GG, D, MEAS, CACHE>(M, c, st);
  KT_EIG_CASE(16, 10, EIG_PLAIN, false)
  KT_EIG_CASE(8, 10, EIG_PLAIN, false)
  KT_EIG_CASE(4, 10, EIG_PLAIN, false)
  KT_EIG_CASE(32, 10, EIG_PLAIN, false)
  KT_EIG_CASE(16, 10, EIG_PLAIN, true)
  KT_EIG_CASE(16, 10, EIG_RATIO, false)
  KT_EIG_CASE(16, 10, EIG_BUILD, false)
  KT_EIG_CASE(16, 10, EIG_MEASURE, true)
  KT_EIG_CASE(32, 36, EIG_PLAIN, false)
  KT_EIG_CASE(16, 36, EIG_PLAIN, false)
  KT_EIG_CASE(8, 36, EIG_PLAIN, false)
  KT_EIG_CASE(32, 36, EIG_PLAIN, true)
  KT_EIG_CASE(32, 36, EIG_RATIO, false)
  KT_EIG_CASE(32, 36, EIG_BUILD, false)
  KT_EIG_CASE(32, 36, EIG_MEASURE, true)
#undef KT_EIG_CASE
  return (int)cudaErrorInvalidValue;
}

}  // namespace kt
