// Multigrid V(1,0) cycle on the 9-point element stencils of k_fevar.cu,
// (sigma M + tau K(a)) u = r per spectral plane: the colour-ordered Gauss-Seidel sweep from
// zero, the residual and its restriction by P^T of one level in one launch, and all small
// levels in another: at 127^2 x 130 planes 46 + 29 us an apply, where running colour by colour
// and level by level took 7 (4 + 2 + 1) launches and 324 us of a GMRES iteration's 800.
// Bound by latency and issue (the planes stay in L2).
//
// Colours are c = (i1 & 1) + 2 (i2 & 1).  Two facts keep a level in one array:
// * After the sweep the equation of a point held when the point was swept, so what is left
//   of it is the part of the neighbours swept later: res_P = -sum_{c(Q) > c(P)} A_PQ u_Q.
//   No right-hand side is needed any more (it is overwritten by u), and the points of the
//   last colour have residual zero.
// * An even row needs only itself (colours 0, 1), an odd row the two even rows beside it
//   (colours 2, 3): a strip of rows is swept from r alone with one odd and one even row of
//   halo on each side, and its columns are whole rows, so there is no halo along x1.
// A row of m points lies in shared memory as its (m + 1) / 2 even columns followed by its odd
// ones: the points of a colour and each of their neighbours are then consecutive.
#include <algorithm>

#include "common.cuh"

namespace pcopt {

namespace {

template <typename Tc>
struct FeCoef {
  const Tc* E;  // element coefficients, (m + 1)^2
  typename Cx<Tc>::t sig;
  Tc mh, tau;  // h^2 / 36
  int m;
};

// rows lo, lo + 1, .. of one level
template <typename C>
struct FeRows {
  C* a;
  int m, lo;
  __device__ __forceinline__ C* row(int i2) const { return a + (i2 - lo) * m; }
};

// the four element coefficients around node (i1, i2)
template <typename Tc>
struct FeQuad {
  Tc SW, SE, NW, NE;
};
template <typename Tc>
__device__ __forceinline__ FeQuad<Tc> fe_quad(const FeCoef<Tc>& f, int i1, int i2) {
  const int me = f.m + 1;
  const Tc* e = f.E + i2 * me + i1;
  return FeQuad<Tc>{__ldg(e), __ldg(e + 1), __ldg(e + me), __ldg(e + me + 1)};
}

template <typename C, typename T>
__device__ __forceinline__ void fe_fma(C& acc, T w, C v) {
  acc.x = fma(w, v.x, acc.x);
  acc.y = fma(w, v.y, acc.y);
}

// A_PQ u_Q summed over some neighbours: mh sigma (4 edges + corners) + tau / 6 ku, with
// ku the stiffness sum times 6 (edges -(two elements), corners -2 (one element))
template <typename Tc>
struct FeSum {
  typename Cx<Tc>::t edges, corners, ku;
  __device__ __forceinline__ FeSum() { edges = corners = ku = czero<Tc>(); }
  __device__ __forceinline__ void edge(Tc e, typename Cx<Tc>::t v) {
    edges = edges + v;
    fe_fma(ku, -e, v);
  }
  __device__ __forceinline__ void corner(Tc e, typename Cx<Tc>::t v) {
    corners = corners + v;
    fe_fma(ku, Tc(-2) * e, v);
  }
  __device__ __forceinline__ typename Cx<Tc>::t value(const FeCoef<Tc>& f) const {
    typename Cx<Tc>::t mu, r;
    mu.x = f.mh * fma(Tc(4), edges.x, corners.x);
    mu.y = f.mh * fma(Tc(4), edges.y, corners.y);
    const Tc t6 = f.tau * (Tc(1) / Tc(6));
    r.x = fma(t6, ku.x, f.sig.x * mu.x - f.sig.y * mu.y);
    r.y = fma(t6, ku.y, f.sig.x * mu.y + f.sig.y * mu.x);
    return r;
  }
};

// u = (r - off) / (sigma 16 mh + tau 2/3 (sum of the four elements))
template <typename Tc>
__device__ __forceinline__ typename Cx<Tc>::t fe_point(const FeCoef<Tc>& f, const FeQuad<Tc>& q,
                                                       typename Cx<Tc>::t r, typename Cx<Tc>::t off) {
  typename Cx<Tc>::t dg;
  dg.x = fma(f.sig.x, Tc(16) * f.mh, f.tau * (Tc(2) / Tc(3)) * (q.SW + q.SE + q.NW + q.NE));
  dg.y = f.sig.y * (Tc(16) * f.mh);
  return cmul(r - off, cinv(dg));
}

// colours 0 and 1 of the even rows in [lo, hi], colours 2 and 3 of the odd ones; a warp takes
// a row (nw warps), its lanes the points of a colour.  Ends with a barrier.
template <typename Tc>
__device__ __forceinline__ void fe_sweep(const FeCoef<Tc>& f, const FeRows<typename Cx<Tc>::t>& A, int lo, int hi,
                                         int warp, int nw, int lane) {
  typedef typename Cx<Tc>::t C;
  const int h = (f.m + 1) / 2;  // even columns; h - 1 odd ones
  for (int y = lo + 2 * warp; y <= hi; y += 2 * nw) {
    C* R = A.row(y);
    for (int t = lane; t < h; t += 32) R[t] = fe_point<Tc>(f, fe_quad(f, 2 * t, y), R[t], czero<Tc>());
    __syncwarp();
    for (int t = lane; t < h - 1; t += 32) {
      const FeQuad<Tc> q = fe_quad(f, 2 * t + 1, y);
      FeSum<Tc> s;
      s.edge(q.SW + q.NW, R[t]);
      s.edge(q.SE + q.NE, R[t + 1]);
      R[h + t] = fe_point<Tc>(f, q, R[h + t], s.value(f));
    }
  }
  __syncthreads();
  for (int y = lo + 1 + 2 * warp; y < hi; y += 2 * nw) {
    C* R = A.row(y);
    const C *S = A.row(y - 1), *N = A.row(y + 1);
    for (int t = lane; t < h; t += 32) {
      const FeQuad<Tc> q = fe_quad(f, 2 * t, y);
      FeSum<Tc> s;
      s.edge(q.SW + q.SE, S[t]);
      s.edge(q.NW + q.NE, N[t]);
      if (t > 0) {
        s.corner(q.SW, S[h + t - 1]);
        s.corner(q.NW, N[h + t - 1]);
      }
      if (t < h - 1) {
        s.corner(q.SE, S[h + t]);
        s.corner(q.NE, N[h + t]);
      }
      R[t] = fe_point<Tc>(f, q, R[t], s.value(f));
    }
    __syncwarp();
    for (int t = lane; t < h - 1; t += 32) {
      const FeQuad<Tc> q = fe_quad(f, 2 * t + 1, y);
      FeSum<Tc> s;
      s.edge(q.SW + q.NW, R[t]);
      s.edge(q.SE + q.NE, R[t + 1]);
      s.edge(q.SW + q.SE, S[h + t]);
      s.edge(q.NW + q.NE, N[h + t]);
      s.corner(q.SW, S[t]);
      s.corner(q.SE, S[t + 1]);
      s.corner(q.NW, N[t]);
      s.corner(q.NE, N[t + 1]);
      R[h + t] = fe_point<Tc>(f, q, R[h + t], s.value(f));
    }
  }
  __syncthreads();
}

// minus the residuals of colours 0, 1 (even rows) and 2 (odd rows) of rows y0..y1 into B
template <typename Tc>
__device__ __forceinline__ void fe_residual(const FeCoef<Tc>& f, const FeRows<typename Cx<Tc>::t>& A,
                                            const FeRows<typename Cx<Tc>::t>& B, int y0, int y1, int warp, int nw,
                                            int lane) {
  typedef typename Cx<Tc>::t C;
  const int h = (f.m + 1) / 2;
  for (int y = y0 + warp; y <= y1; y += nw) {
    const C* R = A.row(y);
    C* O = B.row(y);
    if (y & 1) {
      for (int t = lane; t < h; t += 32) {
        const FeQuad<Tc> q = fe_quad(f, 2 * t, y);
        FeSum<Tc> s;
        if (t > 0) s.edge(q.SW + q.NW, R[h + t - 1]);
        if (t < h - 1) s.edge(q.SE + q.NE, R[h + t]);
        O[t] = s.value(f);
      }
      continue;
    }
    const bool so = y > 0, no = y < f.m - 1;
    const C *S = A.row(so ? y - 1 : y), *N = A.row(no ? y + 1 : y);
    for (int t = lane; t < h; t += 32) {
      const FeQuad<Tc> q = fe_quad(f, 2 * t, y);
      const bool w = t > 0, e = t < h - 1;
      FeSum<Tc> s;
      if (w) s.edge(q.SW + q.NW, R[h + t - 1]);
      if (e) s.edge(q.SE + q.NE, R[h + t]);
      if (so) {
        s.edge(q.SW + q.SE, S[t]);
        if (w) s.corner(q.SW, S[h + t - 1]);
        if (e) s.corner(q.SE, S[h + t]);
      }
      if (no) {
        s.edge(q.NW + q.NE, N[t]);
        if (w) s.corner(q.NW, N[h + t - 1]);
        if (e) s.corner(q.NE, N[h + t]);
      }
      O[t] = s.value(f);
    }
    for (int t = lane; t < h - 1; t += 32) {
      const FeQuad<Tc> q = fe_quad(f, 2 * t + 1, y);
      FeSum<Tc> s;
      if (so) {
        s.edge(q.SW + q.SE, S[h + t]);
        s.corner(q.SW, S[t]);
        s.corner(q.SE, S[t + 1]);
      }
      if (no) {
        s.edge(q.NW + q.NE, N[h + t]);
        s.corner(q.NW, N[t]);
        s.corner(q.NE, N[t + 1]);
      }
      O[h + t] = s.value(f);
    }
  }
}

// P^T of the residual at coarse point (I, J) (weights 1, 1/2, 1/4; the centre's is zero)
template <typename C>
__device__ __forceinline__ C fe_restrict(const FeRows<C>& B, int I, int J) {
  const int h = (B.m + 1) / 2;
  const C *S = B.row(2 * J), *R = B.row(2 * J + 1), *N = B.row(2 * J + 2);
  const C ed = R[I] + R[I + 1] + S[h + I] + N[h + I];
  const C co = S[I] + S[I + 1] + N[I] + N[I + 1];
  C v;  // B holds minus the residual
  v.x = -(co.x * 0.25f + ed.x * 0.5f);
  v.y = -(co.y * 0.25f + ed.y * 0.5f);
  return v;
}

// position of column i1 in a row of m points
__device__ __forceinline__ int fe_col(int i1, int m) { return (i1 >> 1) + ((i1 & 1) ? (m + 1) / 2 : 0); }

// One level: strip of cy coarse rows of plane blockIdx.y (see the file's head)
template <typename Tc>
__global__ void __launch_bounds__(256) fe_down_kernel(const typename Cx<Tc>::t* __restrict__ r,
                                                      typename Cx<Tc>::t* __restrict__ u,
                                                      typename Cx<Tc>::t* __restrict__ rc, const Tc* __restrict__ E,
                                                      const typename Cx<Tc>::t* __restrict__ sigma, int m, Tc h2,
                                                      Tc tau, int cy) {
  typedef typename Cx<Tc>::t C;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int p = blockIdx.y, mc = (m - 1) / 2;
  const int J0 = blockIdx.x * cy, J1 = min(mc, J0 + cy);  // coarse rows [J0, J1)
  const int lo = max(0, 2 * J0 - 2), hi = min(m - 1, 2 * J1 + 2);
  const FeRows<C> A{reinterpret_cast<C*>(smem_raw), m, lo};
  const FeRows<C> B{A.a + (hi - lo + 1) * m, m, 2 * J0};
  const FeCoef<Tc> f{E, sigma[p], h2 / Tc(36), tau, m};
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
  const int64_t base = (int64_t)p * m * m;
  for (int y = lo + warp; y <= hi; y += nw)
    for (int i1 = lane; i1 < m; i1 += 32) A.row(y)[fe_col(i1, m)] = r[base + (int64_t)y * m + i1];
  __syncthreads();
  fe_sweep<Tc>(f, A, lo, hi, warp, nw, lane);
  fe_residual<Tc>(f, A, B, 2 * J0, 2 * J1, warp, nw, lane);
  const int y1 = J1 == mc ? m : 2 * J1;  // the strip's own rows
  for (int y = 2 * J0 + warp; y < y1; y += nw)
    for (int i1 = lane; i1 < m; i1 += 32) u[base + (int64_t)y * m + i1] = A.row(y)[fe_col(i1, m)];
  __syncthreads();
  for (int J = J0 + warp; J < J1; J += nw)
    for (int I = lane; I < mc; I += 32) rc[((int64_t)p * mc + J) * mc + I] = fe_restrict(B, I, J);
}

// Every level from lv.m[0] down to the one-point level and back, one CTA a plane
constexpr int kFeTailThreads = 512;
template <typename Tc>
__global__ void __launch_bounds__(kFeTailThreads) fe_tail_kernel(FeLevels<Tc> lv,
                                                                 const typename Cx<Tc>::t* __restrict__ r0,
                                                                 typename Cx<Tc>::t* __restrict__ u0,
                                                                 const typename Cx<Tc>::t* __restrict__ sigma,
                                                                 Tc tau) {
  typedef typename Cx<Tc>::t C;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C* A[kMaxCoarseLevels];
  C* q = reinterpret_cast<C*>(smem_raw);
  for (int l = 0; l < lv.count; ++l) {
    A[l] = q;
    q += lv.m[l] * lv.m[l];
  }
  C* const res = q;  // minus the residual of one level
  const int p = blockIdx.x, m0 = lv.m[0];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = kFeTailThreads / 32;
  const C sig = sigma[p];
  const int64_t base = (int64_t)p * m0 * m0;
  for (int y = warp; y < m0; y += nw)
    for (int i1 = lane; i1 < m0; i1 += 32) A[0][y * m0 + fe_col(i1, m0)] = r0[base + y * m0 + i1];
  __syncthreads();
  for (int l = 0; l < lv.count; ++l) {
    const int m = lv.m[l];
    const Tc hl = Tc(1) / Tc(m + 1);
    const FeCoef<Tc> f{lv.E[l], sig, hl * hl / Tc(36), tau, m};
    const FeRows<C> R{A[l], m, 0};
    fe_sweep<Tc>(f, R, 0, m - 1, warp, nw, lane);
    if (l + 1 == lv.count) break;  // the one-point level is solved by its sweep
    const FeRows<C> B{res, m, 0};
    fe_residual<Tc>(f, R, B, 0, m - 1, warp, nw, lane);
    __syncthreads();
    const int mc = lv.m[l + 1];
    for (int J = warp; J < mc; J += nw)
      for (int I = lane; I < mc; I += 32) A[l + 1][J * mc + fe_col(I, mc)] = fe_restrict(B, I, J);
    __syncthreads();
  }
  // up: u_l += P u_{l+1}; coarse point (I, J) sits on the odd columns and rows
  for (int l = lv.count - 2; l >= 0; --l) {
    const int m = lv.m[l], mc = lv.m[l + 1], h = (m + 1) / 2;
    auto coarse = [&](int I, int J) -> C {
      return I >= 0 && I < mc && J >= 0 && J < mc ? A[l + 1][J * mc + fe_col(I, mc)] : czero<Tc>();
    };
    for (int y = warp; y < m; y += nw) {
      C* R = A[l] + y * m;
      const int J = y >> 1;  // odd rows sit on coarse row J, even ones between J - 1 and J
      for (int t = lane; t < h; t += 32) {
        const C e1 = coarse(t, J), e0 = coarse(t - 1, J);
        C ev = e0 + e1, od = e1;
        Tc we = Tc(0.5), wo = Tc(1);
        if (!(y & 1)) {
          const C b1 = coarse(t, J - 1), b0 = coarse(t - 1, J - 1);
          ev = ev + b0 + b1;
          od = od + b1;
          we = Tc(0.25);
          wo = Tc(0.5);
        }
        fe_fma(R[t], we, ev);
        if (t < h - 1) fe_fma(R[h + t], wo, od);
      }
    }
    __syncthreads();
  }
  for (int y = warp; y < m0; y += nw)
    for (int i1 = lane; i1 < m0; i1 += 32) u0[base + y * m0 + i1] = A[0][y * m0 + fe_col(i1, m0)];
}

constexpr size_t kFeSmem = 227 * 1024;

template <typename Tc>
size_t fe_down_smem(int m, int cy) {
  return sizeof(typename Cx<Tc>::t) * (size_t)m * ((2 * cy + 5) + (2 * cy + 1));
}

}  // namespace

// coarse rows per strip: 1.0 + 2.5 / cy of the sweep's work is done, so the longest strip that
// leaves three CTAs an SM and fills the chip twice; 0 where not even one row fits
template <typename Tc>
int fe_down_rows(int m, int planes) {
  const int mc = (m - 1) / 2;
  if (mc < 1 || fe_down_smem<Tc>(m, 1) > kFeSmem) return 0;
  int cy = 16;
  while (cy > 1 && (fe_down_smem<Tc>(m, cy) > 72 * 1024 ||
                    (cy > 4 && (int64_t)planes * ((mc + cy - 1) / cy) < 2 * num_sms())))
    cy >>= 1;
  return cy;
}

template <typename Tc>
cudaError_t launch_fe_down(Launch& L, int m, int planes, Tc h2, Tc tau, const Tc* E, const typename Cx<Tc>::t* sigma,
                           const typename Cx<Tc>::t* r, typename Cx<Tc>::t* u, typename Cx<Tc>::t* rc) {
  const int cy = fe_down_rows<Tc>(m, planes), mc = (m - 1) / 2;
  if (cy < 1) return cudaErrorInvalidValue;
  const size_t smem = fe_down_smem<Tc>(m, cy);
  cudaError_t e = allow_dynamic_smem(fe_down_kernel<Tc>, smem);
  if (e != cudaSuccess) return e;
  const double cs = sizeof(typename Cx<Tc>::t), np = (double)m * m * planes;
  L.begin(KC_MG_DOWN);
  fe_down_kernel<Tc><<<dim3((unsigned)((mc + cy - 1) / cy), (unsigned)planes), 256, smem, L.stream>>>(
      r, u, rc, E, sigma, m, h2, tau, cy);
  return L.end(KC_MG_DOWN, np * 2.25 * cs, np * 80.0);
}

template <typename Tc>
size_t fe_tail_smem(const FeLevels<Tc>& lv) {
  size_t n = (size_t)lv.m[0] * lv.m[0];
  for (int l = 0; l < lv.count; ++l) n += (size_t)lv.m[l] * lv.m[l];
  return n * sizeof(typename Cx<Tc>::t);
}

template <typename Tc>
cudaError_t launch_fe_tail(Launch& L, int planes, const FeLevels<Tc>& lv, Tc tau, const typename Cx<Tc>::t* sigma,
                           const typename Cx<Tc>::t* r, typename Cx<Tc>::t* u) {
  const size_t smem = fe_tail_smem(lv);
  cudaError_t e = allow_dynamic_smem(fe_tail_kernel<Tc>, smem);
  if (e != cudaSuccess) return e;
  const double cs = sizeof(typename Cx<Tc>::t), np = (double)lv.m[0] * lv.m[0] * planes;
  L.begin(KC_MG_COARSE);
  fe_tail_kernel<Tc><<<(unsigned)planes, kFeTailThreads, smem, L.stream>>>(lv, r, u, sigma, tau);
  return L.end(KC_MG_COARSE, 2.0 * np * cs, 100.0 * np);
}

#define PCOPT_FEMG(Tc)                                                                                         \
  template int fe_down_rows<Tc>(int, int);                                                                     \
  template cudaError_t launch_fe_down<Tc>(Launch&, int, int, Tc, Tc, const Tc*, const Cx<Tc>::t*,              \
                                          const Cx<Tc>::t*, Cx<Tc>::t*, Cx<Tc>::t*);                           \
  template cudaError_t launch_fe_tail<Tc>(Launch&, int, const FeLevels<Tc>&, Tc, const Cx<Tc>::t*,             \
                                          const Cx<Tc>::t*, Cx<Tc>::t*);
PCOPT_FEMG(float)
PCOPT_FEMG(double)
#undef PCOPT_FEMG

}  // namespace pcopt
