// The finest multigrid correction as the inverse time transforms apply it (FineCorrection).
#pragma once

#include "common.cuh"

namespace pcopt {

// Parents of fine point s in the next coarser level and their linear weights,
// per axis: odd f sits on coarse point (f-1)/2 (weight 1), even f halfway between
// f/2-1 and f/2 (1/2 each, a parent outside [0, mc) is the zero boundary).
template <typename Tc, typename TU>
struct Parents {
  int o[3][2];
  Tc wt[3][2];
  __device__ __forceinline__ void init(const FineCorrection<TU>& fc, int64_t s) {
    int f[3];
    f[0] = (int)(s % fc.mf);
    const int64_t r = s / fc.mf;
    f[1] = (int)(fc.dim == 2 ? r : r % fc.mf);
    f[2] = fc.dim == 3 ? (int)(r / fc.mf) : 0;
    int stride = 1;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      if (a >= fc.dim) {
        o[a][0] = o[a][1] = 0;
        wt[a][0] = Tc(1);
        wt[a][1] = Tc(0);
        continue;
      }
      if (f[a] & 1) {
        o[a][0] = o[a][1] = ((f[a] - 1) >> 1) * stride;
        wt[a][0] = Tc(1);
        wt[a][1] = Tc(0);
      } else {
        int lo = (f[a] >> 1) - 1, hi = f[a] >> 1;
        wt[a][0] = lo >= 0 ? Tc(0.5) : Tc(0);
        wt[a][1] = hi < fc.mc ? Tc(0.5) : Tc(0);
        if (lo < 0) lo = hi;
        if (hi >= fc.mc) hi = lo;
        o[a][0] = lo * stride;
        o[a][1] = hi * stride;
      }
      stride *= fc.mc;
    }
  }
  __device__ __forceinline__ typename Cx<Tc>::t at(const FineCorrection<TU>& fc, int p) const {
    typedef typename Cx<Tc>::t C;
    const TU* e = fc.ec + (int64_t)p * fc.npc;
    C acc = czero<Tc>();
    for (int c2 = 0; c2 < (fc.dim == 3 ? 2 : 1); ++c2)
#pragma unroll
      for (int c1 = 0; c1 < 2; ++c1)
#pragma unroll
        for (int c0 = 0; c0 < 2; ++c0) {
          const Tc w = wt[2][c2] * wt[1][c1] * wt[0][c0];
          if (w != Tc(0)) {
            const C v = ldc(e, o[2][c2] + o[1][c1] + o[0][c0]);
            acc.x = fma(w, v.x, acc.x);
            acc.y = fma(w, v.y, acc.y);
          }
        }
    return acc;
  }
};

}  // namespace pcopt
