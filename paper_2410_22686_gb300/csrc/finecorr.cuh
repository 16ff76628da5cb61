// The finest multigrid correction as the inverse time transforms apply it (FineCorrection).
#pragma once

#include "common.cuh"

namespace pcopt {

// Parents of fine point s in the next coarser level of a 2D grid, per axis: odd f sits on
// coarse point (f-1)/2 (weight 1), even f halfway between f/2-1 and f/2 (1/2 each, a parent
// outside [0, mc) is the zero boundary).  All parents of a point have the same weight, so
// their sum, in grid order, is scaled once: a power of two, so exactly as if each were.
template <typename Tc, typename TU>
struct Parents {
  int o[4];  // coarse offsets, -1: none
  Tc wt;
  __device__ __forceinline__ void init(const FineCorrection<TU>& fc, int64_t s) {
    const int f2 = (int)(s / fc.mf), f1 = (int)(s - (int64_t)f2 * fc.mf);
    const int x1 = f1 >> 1, y1 = f2 >> 1;
    const int x0 = (f1 & 1) ? -1 : x1 - 1, y0 = (f2 & 1) ? -1 : y1 - 1;
    const bool bx = x1 < fc.mc, by = y1 < fc.mc;
    o[0] = x0 >= 0 && y0 >= 0 ? y0 * fc.mc + x0 : -1;
    o[1] = bx && y0 >= 0 ? y0 * fc.mc + x1 : -1;
    o[2] = x0 >= 0 && by ? y1 * fc.mc + x0 : -1;
    o[3] = bx && by ? y1 * fc.mc + x1 : -1;
    wt = ((f1 & 1) ? Tc(1) : Tc(0.5)) * ((f2 & 1) ? Tc(1) : Tc(0.5));
  }
  // v + (P e_c) of plane p
  __device__ __forceinline__ typename Cx<Tc>::t corrected(typename Cx<Tc>::t v, const FineCorrection<TU>& fc,
                                                          int p) const {
    typedef typename Cx<Tc>::t C;
    const TU* e = fc.ec + (int64_t)p * fc.npc;
    C acc = czero<Tc>();
#pragma unroll
    for (int q = 0; q < 4; ++q)
      if (o[q] >= 0) acc = acc + ldc(e, o[q]);
    v.x = fma(wt, acc.x, v.x);
    v.y = fma(wt, acc.y, v.y);
    return v;
  }
};

}  // namespace pcopt
