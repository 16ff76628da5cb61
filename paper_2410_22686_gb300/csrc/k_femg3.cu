// The element multigrid cycle in 3D (27-point stencils of k_fevar3.cu), the counterpart of
// k_femg.cu: colours c = (i1 & 1) + 2 (i2 & 1) + 4 (i3 & 1), the sweep from zero kept in one
// array, the residual formed from the neighbours swept later.
//
// Rows of one parity (i2, i3) need only rows of the parities before them: even layers
// (colours 0..3) are independent of each other, and an odd layer needs the two even ones
// beside it.  A fine level takes three launches: even layers, odd layers (a strip of rows of
// one layer per CTA, swept in shared memory), and residual + restriction by P^T (a strip of
// coarse rows of one coarse layer).  The levels from 15^3 down and back take one launch, a
// CTA per plane.  At 31^3 x 66 planes an apply takes 48 (layers) + 68
// (residual and restriction) + 53 us (lower levels); colour by colour and level by level it
// was 49 launches and 424 us of a GMRES iteration's 740.  Bound by latency and issue.
// Rows lie in shared memory as in k_femg.cu: even columns, then odd ones.
#include <algorithm>

#include "common.cuh"

namespace pcopt {

namespace {

constexpr int kFe3Threads = 256;

template <int V>
struct Fe3Int {
  static constexpr int value = V;
};

template <typename Tc>
struct Fe3Coef {
  const Tc* E;  // element coefficients, (m + 1)^3
  typename Cx<Tc>::t sig;
  Tc mh, tk;  // h^3 / 216, tau h / 12
  int m;
};

__device__ __forceinline__ int fe3_col(int i1, int m) { return (i1 >> 1) + ((i1 & 1) ? (m + 1) / 2 : 0); }

// lanes that share a row: the smallest power of two >= its (m + 1) / 2 even columns, 4..32
__host__ __device__ __forceinline__ int fe3_lanes(int m) { return m > 31 ? 32 : m > 15 ? 16 : m > 7 ? 8 : 4; }

// rows y, z around the one in hand; row(o2, o3) of it (called for existing rows only)
template <typename C>
struct Fe3At {
  C* a;           // row (y, z)
  int sy, sz;     // distance of rows y + 1 and z + 1
  bool y0, y1, z0, z1;  // whether y - 1, y + 1, z - 1, z + 1 exist
  __device__ __forceinline__ C* row(int o2, int o3) const { return a + o2 * sy + o3 * sz; }
  __device__ __forceinline__ bool has(int o2, int o3) const {
    return (o2 == 0 || (o2 < 0 ? y0 : y1)) && (o3 == 0 || (o3 < 0 ? z0 : z1));
  }
};

// the eight elements around a node: A[c] holds it at corner c = c1 + 2 c2 + 4 c3
template <typename Tc>
__device__ __forceinline__ void fe3_around(const Fe3Coef<Tc>& f, int i1, int i2, int i3, Tc (&A)[8]) {
  const int me = f.m + 1;
  const Tc* e = f.E + ((int64_t)i3 * me + i2) * me + i1;
#pragma unroll
  for (int c = 0; c < 8; ++c)
    A[c] = __ldg(e + (1 - (c & 1)) + (1 - ((c >> 1) & 1)) * me + (int64_t)(1 - (c >> 2)) * me * me);
}

// sum over the neighbours Q of a point of colour COL (its column index among its parity: t)
// with a lower (HIGH: higher) colour of A_PQ u_Q
template <typename Tc, int COL, bool HIGH>
__device__ __forceinline__ typename Cx<Tc>::t fe3_sum(const Fe3Coef<Tc>& f, const Fe3At<typename Cx<Tc>::t>& at,
                                                      const Tc (&A)[8], int t) {
  typedef typename Cx<Tc>::t C;
  constexpr int px = COL & 1, py = (COL >> 1) & 1, pz = COL >> 2;
  const int h = (f.m + 1) / 2;
  C face = czero<Tc>(), edge = czero<Tc>(), corn = czero<Tc>(), ku = czero<Tc>();
#pragma unroll
  for (int o3 = -1; o3 <= 1; ++o3)
#pragma unroll
    for (int o2 = -1; o2 <= 1; ++o2) {
      const int rc = 2 * (py ^ (o2 & 1)) + 4 * (pz ^ (o3 & 1));  // the row's colours: rc, rc + 1
      if (HIGH ? rc + 1 <= COL : rc >= COL) continue;
      if ((py == 0 || pz == 0) && !at.has(o2, o3)) continue;
      const C* R = at.row(o2, o3);
#pragma unroll
      for (int o1 = -1; o1 <= 1; ++o1) {
        const int nc = rc + (px ^ (o1 & 1)), k = (o1 != 0) + (o2 != 0) + (o3 != 0);
        if (k == 0 || (HIGH ? nc <= COL : nc >= COL)) continue;
        if (px == 0 && o1 != 0 && (o1 < 0 ? t == 0 : t == h - 1)) continue;
        // even column t: odd columns t - 1, t beside it; odd column t: even columns t, t + 1
        const int i = px == 0 ? (o1 == 0 ? t : h + t + (o1 < 0 ? -1 : 0)) : (o1 == 0 ? h + t : t + (o1 < 0 ? 0 : 1));
        const C v = R[i];
        if (k == 1) {
          face = face + v;
          continue;
        }
        Tc s = Tc(0);
#pragma unroll
        for (int c = 0; c < 8; ++c)  // the elements that hold both points
          if ((o1 == 0 || (c & 1) == (o1 < 0)) && (o2 == 0 || ((c >> 1) & 1) == (o2 < 0)) &&
              (o3 == 0 || (c >> 2) == (o3 < 0)))
            s += A[c];
        ku.x = fma(-s, v.x, ku.x);
        ku.y = fma(-s, v.y, ku.y);
        if (k == 2)
          edge = edge + v;
        else
          corn = corn + v;
      }
    }
  C mu, r;
  mu.x = f.mh * fma(Tc(16), face.x, fma(Tc(4), edge.x, corn.x));
  mu.y = f.mh * fma(Tc(16), face.y, fma(Tc(4), edge.y, corn.y));
  r.x = fma(f.tk, ku.x, f.sig.x * mu.x - f.sig.y * mu.y);
  r.y = fma(f.tk, ku.y, f.sig.x * mu.y + f.sig.y * mu.x);
  return r;
}

// u = (r - off) / (64 mh sigma + 4 tk sum of the eight elements)
template <typename Tc>
__device__ __forceinline__ typename Cx<Tc>::t fe3_point(const Fe3Coef<Tc>& f, const Tc (&A)[8],
                                                        typename Cx<Tc>::t r, typename Cx<Tc>::t off) {
  typename Cx<Tc>::t dg;
  const Tc s = ((A[0] + A[1]) + (A[2] + A[3])) + ((A[4] + A[5]) + (A[6] + A[7]));
  dg.x = fma(f.sig.x, Tc(64) * f.mh, Tc(4) * f.tk * s);
  dg.y = f.sig.y * (Tc(64) * f.mh);
  return cmul(r - off, cinv(dg));
}

// both colours of one row (parity PY, PZ) by a group of G lanes; every lane of the warp calls
// it (`on`: the group has a row)
template <typename Tc, int PY, int PZ>
__device__ __forceinline__ void fe3_sweep_row(const Fe3Coef<Tc>& f, const Fe3At<typename Cx<Tc>::t>& at, int y, int z,
                                              bool on, int lane, int G) {
  constexpr int COL = 2 * PY + 4 * PZ;
  const int h = (f.m + 1) / 2;
  if (on)
    for (int t = lane; t < h; t += G) {
      Tc A[8];
      fe3_around(f, 2 * t, y, z, A);
      at.a[t] = fe3_point<Tc>(f, A, at.a[t], fe3_sum<Tc, COL, false>(f, at, A, t));
    }
  __syncwarp();
  if (on)
    for (int t = lane; t < h - 1; t += G) {
      Tc A[8];
      fe3_around(f, 2 * t + 1, y, z, A);
      at.a[h + t] = fe3_point<Tc>(f, A, at.a[h + t], fe3_sum<Tc, COL + 1, false>(f, at, A, t));
    }
}

// minus the residual of one row's points into O (the last colour's is zero and not written)
template <typename Tc, int PY, int PZ>
__device__ __forceinline__ void fe3_residual_row(const Fe3Coef<Tc>& f, const Fe3At<typename Cx<Tc>::t>& at,
                                                 typename Cx<Tc>::t* O, int y, int z, int lane, int G) {
  constexpr int COL = 2 * PY + 4 * PZ;
  const int h = (f.m + 1) / 2;
  for (int t = lane; t < h; t += G) {
    Tc A[8];
    fe3_around(f, 2 * t, y, z, A);
    O[t] = fe3_sum<Tc, COL, true>(f, at, A, t);
  }
  if (COL + 1 == 7) return;
  for (int t = lane; t < h - 1; t += G) {
    Tc A[8];
    fe3_around(f, 2 * t + 1, y, z, A);
    O[h + t] = fe3_sum<Tc, (COL + 1) & 7, true>(f, at, A, t);
  }
}

template <typename Tc>
__device__ __forceinline__ void fe3_residual_any(const Fe3Coef<Tc>& f, const Fe3At<typename Cx<Tc>::t>& at,
                                                 typename Cx<Tc>::t* O, int y, int z, int lane, int G) {
  if (z & 1) {
    if (y & 1)
      fe3_residual_row<Tc, 1, 1>(f, at, O, y, z, lane, G);
    else
      fe3_residual_row<Tc, 0, 1>(f, at, O, y, z, lane, G);
  } else if (y & 1) {
    fe3_residual_row<Tc, 1, 0>(f, at, O, y, z, lane, G);
  } else {
    fe3_residual_row<Tc, 0, 0>(f, at, O, y, z, lane, G);
  }
}

// P^T at coarse column I from minus the residual's rows: row(o2, o3) is the fine row beside
// the coarse point's (weights 1/2 per coordinate off it; the point's own residual is zero)
template <typename Tc, typename Row>
__device__ __forceinline__ typename Cx<Tc>::t fe3_restrict(Row row, int I, int h) {
  typedef typename Cx<Tc>::t C;
  C acc = czero<Tc>();
#pragma unroll
  for (int o3 = -1; o3 <= 1; ++o3)
#pragma unroll
    for (int o2 = -1; o2 <= 1; ++o2) {
      const C* R = row(o2, o3);
      const Tc w = -(o2 == 0 ? Tc(1) : Tc(0.5)) * (o3 == 0 ? Tc(1) : Tc(0.5));
      C v = R[I] + R[I + 1];
      v.x *= Tc(0.5);
      v.y *= Tc(0.5);
      if (o2 != 0 || o3 != 0) v = v + R[h + I];
      acc.x = fma(w, v.x, acc.x);
      acc.y = fma(w, v.y, acc.y);
    }
  return acc;
}

// Rows 2 Y0 .. 2 Y0 + 2 cy of one layer of plane blockIdx.z: the even ones from themselves (and,
// in an odd layer, the layers beside it), the odd ones from the even ones; all but the last
// even row belong to the strip (the level's last row too).
template <typename Tc, int PZ>
__global__ void __launch_bounds__(kFe3Threads) fe3_layer_kernel(const typename Cx<Tc>::t* __restrict__ r,
                                                                typename Cx<Tc>::t* __restrict__ u,
                                                                const Tc* __restrict__ E,
                                                                const typename Cx<Tc>::t* __restrict__ sigma, int m,
                                                                Tc h, Tc tau, int cy) {
  typedef typename Cx<Tc>::t C;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int z = 2 * blockIdx.y + PZ, p = blockIdx.z;
  const int Y0 = 2 * blockIdx.x * cy, Y1 = min(m - 1, Y0 + 2 * cy);  // even rows Y0, .., Y1
  const int nr = Y1 - Y0 + 3;  // rows Y0 - 1 .. Y1 + 1 of a layer in shared memory
  // layers z - 1, z, z + 1 (PZ = 0: z alone); row y of layer z at buf + (y - Y0 + 1) m
  C* const buf = reinterpret_cast<C*>(smem_raw) + (PZ ? nr * m : 0);
  const Fe3Coef<Tc> f{E, sigma[p], h * h * h / Tc(216), tau * h / Tc(12), m};
  const int G = fe3_lanes(m), per = 32 / G, nw = kFe3Threads / 32;
  const int warp = threadIdx.x >> 5, lane = (threadIdx.x & 31) & (G - 1), sub = (threadIdx.x & 31) / G;
  const int64_t lay = (int64_t)m * m, base = (int64_t)p * m * lay;
  if (PZ) {
    for (int k = warp * per + sub; k < 2 * nr; k += nw * per) {
      const int side = k < nr ? 0 : 1, y = Y0 - 1 + (k - side * nr);
      if (y < 0 || y >= m) continue;
      const C* src = u + base + (int64_t)(z - 1 + 2 * side) * lay + (int64_t)y * m;
      C* dst = buf + (side ? 1 : -1) * nr * m + (y - Y0 + 1) * m;
      for (int i = lane; i < m; i += G) dst[fe3_col(i, m)] = src[i];
    }
  }
  for (int y = Y0 + warp * per + sub; y <= Y1; y += nw * per) {
    const C* src = r + base + (int64_t)z * lay + (int64_t)y * m;
    for (int i = lane; i < m; i += G) buf[(y - Y0 + 1) * m + fe3_col(i, m)] = src[i];
  }
  __syncthreads();
  const bool zz = PZ != 0;
  for (int k = warp * per; Y0 + 2 * k <= Y1; k += nw * per) {
    const int y = Y0 + 2 * (k + sub);
    const Fe3At<C> at{buf + (y - Y0 + 1) * m, m, nr * m, y > 0, y < m - 1, zz, zz};
    fe3_sweep_row<Tc, 0, PZ>(f, at, y, z, y <= Y1, lane, G);
  }
  __syncthreads();
  for (int k = warp * per; Y0 + 1 + 2 * k < Y1; k += nw * per) {
    const int y = Y0 + 1 + 2 * (k + sub);
    const Fe3At<C> at{buf + (y - Y0 + 1) * m, m, nr * m, true, true, zz, zz};
    fe3_sweep_row<Tc, 1, PZ>(f, at, y, z, y < Y1, lane, G);
  }
  __syncthreads();
  const int yl = Y1 == m - 1 ? Y1 : Y1 - 1;
  for (int y = Y0 + warp * per + sub; y <= yl; y += nw * per) {
    C* dst = u + base + (int64_t)z * lay + (int64_t)y * m;
    for (int i = lane; i < m; i += G) dst[i] = buf[(y - Y0 + 1) * m + fe3_col(i, m)];
  }
}

// coarse rows J0 .. J0 + cy - 1 of coarse layer blockIdx.y of plane blockIdx.z
template <typename Tc>
__global__ void __launch_bounds__(kFe3Threads) fe3_restrict_kernel(const typename Cx<Tc>::t* __restrict__ u,
                                                                   typename Cx<Tc>::t* __restrict__ rc,
                                                                   const Tc* __restrict__ E,
                                                                   const typename Cx<Tc>::t* __restrict__ sigma, int m,
                                                                   Tc h, Tc tau, int cy) {
  typedef typename Cx<Tc>::t C;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int K = blockIdx.y, p = blockIdx.z, mc = (m - 1) / 2, hm = (m + 1) / 2;
  const int J0 = blockIdx.x * cy, J1 = min(mc, J0 + cy);
  const int nu = 2 * cy + 3, nres = 2 * cy + 1;  // rows of u (from 2 J0 - 1) and of the residual (from 2 J0)
  C* const U = reinterpret_cast<C*>(smem_raw);  // [5][nu][m]: layers 2K - 1 .. 2K + 3
  C* const R = U + 5 * nu * m;                  // [3][nres][m]: layers 2K .. 2K + 2
  const Fe3Coef<Tc> f{E, sigma[p], h * h * h / Tc(216), tau * h / Tc(12), m};
  const int G = fe3_lanes(m), per = 32 / G, nw = kFe3Threads / 32;
  const int warp = threadIdx.x >> 5, lane = (threadIdx.x & 31) & (G - 1), sub = (threadIdx.x & 31) / G;
  const int64_t lay = (int64_t)m * m, base = (int64_t)p * m * lay;
  for (int k = warp * per + sub; k < 5 * nu; k += nw * per) {
    const int q = k / nu, z = 2 * K - 1 + q, y = 2 * J0 - 1 + (k - q * nu);
    if (z < 0 || z >= m || y < 0 || y >= m) continue;
    const C* src = u + base + (int64_t)z * lay + (int64_t)y * m;
    for (int i = lane; i < m; i += G) U[k * m + fe3_col(i, m)] = src[i];
  }
  __syncthreads();
  for (int k = warp * per + sub; k < 3 * nres; k += nw * per) {
    const int q = k / nres, z = 2 * K + q, y = 2 * J0 + (k - q * nres);
    if (y > 2 * J1) continue;
    const Fe3At<C> at{U + ((q + 1) * nu + (y - 2 * J0 + 1)) * m, m, nu * m, y > 0, y < m - 1, z > 0, z < m - 1};
    fe3_residual_any<Tc>(f, at, R + k * m, y, z, lane, G);
  }
  __syncthreads();
  const int n = (J1 - J0) * mc;
  for (int e = threadIdx.x; e < n; e += kFe3Threads) {
    const int j = e / mc, I = e - j * mc;
    auto row = [&](int o2, int o3) -> const C* { return R + ((1 + o3) * nres + 2 * j + 1 + o2) * m; };
    rc[(((int64_t)p * mc + K) * mc + J0 + j) * mc + I] = fe3_restrict<Tc>(row, I, hm);
  }
}

// Every level from lv.m[0] <= 15 down to the one-point level and back, one CTA a plane
constexpr int kFe3TailThreads = 512;
template <typename Tc>
__global__ void __launch_bounds__(kFe3TailThreads) fe3_tail_kernel(FeLevels<Tc> lv,
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
    q += lv.m[l] * lv.m[l] * lv.m[l];
  }
  C* const res = q;  // minus the residual of one level
  const int p = blockIdx.x, m0 = lv.m[0], np0 = m0 * m0 * m0;
  const int warp = threadIdx.x >> 5, wl = threadIdx.x & 31, nw = kFe3TailThreads / 32;
  const C sig = sigma[p];
  for (int e = threadIdx.x; e < np0; e += kFe3TailThreads) {
    const int y = e / m0, i = e - y * m0;
    A[0][y * m0 + fe3_col(i, m0)] = r0[(int64_t)p * np0 + e];
  }
  __syncthreads();
  for (int l = 0; l < lv.count; ++l) {
    const int m = lv.m[l], h = (m + 1) / 2;
    const Tc hl = Tc(1) / Tc(m + 1);
    const Fe3Coef<Tc> f{lv.E[l], sig, hl * hl * hl / Tc(216), tau * hl / Tc(12), m};
    const int G = fe3_lanes(m), per = 32 / G, lane = wl & (G - 1), sub = wl / G;
    // the rows of parity (py, pz), ny x nz of them, in this order
    auto phase = [&](auto PYc, auto PZc) {
      constexpr int PY = decltype(PYc)::value, PZ = decltype(PZc)::value;
      const int ny = PY ? h - 1 : h, nz = PZ ? h - 1 : h;
      for (int k = warp * per; k < ny * nz; k += nw * per) {
        const int kk = k + sub;
        const int z = 2 * (kk / ny) + PZ, y = 2 * (kk % ny) + PY;
        const bool on = kk < ny * nz;
        const Fe3At<C> at{A[l] + (on ? (z * m + y) * m : 0), m, m * m, y > 0, y < m - 1, z > 0, z < m - 1};
        fe3_sweep_row<Tc, PY, PZ>(f, at, y, z, on, lane, G);
      }
      __syncthreads();
    };
    phase(Fe3Int<0>(), Fe3Int<0>());
    if (m > 1) {
      phase(Fe3Int<1>(), Fe3Int<0>());
      phase(Fe3Int<0>(), Fe3Int<1>());
      phase(Fe3Int<1>(), Fe3Int<1>());
    }
    if (l + 1 == lv.count) break;  // the one-point level is solved by its sweep
    for (int k = warp * per + sub; k < m * m; k += nw * per) {
      const int z = k / m, y = k - z * m;
      const Fe3At<C> at{A[l] + k * m, m, m * m, y > 0, y < m - 1, z > 0, z < m - 1};
      fe3_residual_any<Tc>(f, at, res + k * m, y, z, lane, G);
    }
    __syncthreads();
    const int mc = lv.m[l + 1];
    for (int e = threadIdx.x; e < mc * mc * mc; e += kFe3TailThreads) {
      const int I = e % mc, JK = e / mc, J = JK % mc, K = JK / mc;
      auto row = [&](int o2, int o3) -> const C* { return res + ((2 * K + 1 + o3) * m + 2 * J + 1 + o2) * m; };
      A[l + 1][JK * mc + fe3_col(I, mc)] = fe3_restrict<Tc>(row, I, h);
    }
    __syncthreads();
  }
  // up: u_l += P u_{l+1}; coarse point I sits on the odd column 2 I + 1
  for (int l = lv.count - 2; l >= 0; --l) {
    const int m = lv.m[l], mc = lv.m[l + 1];
    for (int e = threadIdx.x; e < m * m * m; e += kFe3TailThreads) {
      const int i1 = e % m, yz = e / m, i2 = yz % m, i3 = yz / m;
      C acc = czero<Tc>();
#pragma unroll
      for (int c = 0; c < 8; ++c) {
        // parents I = i / 2 (both parities) and, for an even index, i / 2 - 1
        const int d1 = c & 1, d2 = (c >> 1) & 1, d3 = c >> 2;
        const int I = (i1 >> 1) - d1, J = (i2 >> 1) - d2, K = (i3 >> 1) - d3;
        if ((d1 && (i1 & 1)) || (d2 && (i2 & 1)) || (d3 && (i3 & 1))) continue;
        if (I < 0 || I >= mc || J < 0 || J >= mc || K < 0 || K >= mc) continue;
        acc = acc + A[l + 1][(K * mc + J) * mc + fe3_col(I, mc)];
      }
      const Tc w = ((i1 & 1) ? Tc(1) : Tc(0.5)) * ((i2 & 1) ? Tc(1) : Tc(0.5)) * ((i3 & 1) ? Tc(1) : Tc(0.5));
      C& d = A[l][yz * m + fe3_col(i1, m)];
      d.x = fma(w, acc.x, d.x);
      d.y = fma(w, acc.y, d.y);
    }
    __syncthreads();
  }
  for (int e = threadIdx.x; e < np0; e += kFe3TailThreads) {
    const int y = e / m0, i = e - y * m0;
    u0[(int64_t)p * np0 + e] = A[0][y * m0 + fe3_col(i, m0)];
  }
}

constexpr size_t kFe3Smem = 227 * 1024;

template <typename Tc>
size_t fe3_odd_smem(int m, int cy) {
  return sizeof(typename Cx<Tc>::t) * (size_t)m * 3 * (2 * cy + 3);
}
template <typename Tc>
size_t fe3_restrict_smem(int m, int cy) {
  return sizeof(typename Cx<Tc>::t) * (size_t)m * (5 * (2 * cy + 3) + 3 * (2 * cy + 1));
}

// the longest strip (row pairs or coarse rows) of up to `most` that leaves four CTAs an SM
template <typename F>
int fe3_longest(int m, int most, F smem) {
  int cy = 1;
  while (2 * cy <= most && cy < (m + 1) / 2 && smem(m, 2 * cy) <= 56 * 1024) cy *= 2;
  return cy;
}

}  // namespace

template <typename Tc>
bool fe3_down_fits(int m) {
  return m >= 3 && fe3_restrict_smem<Tc>(m, 1) <= kFe3Smem && m < 65536;
}

template <typename Tc>
cudaError_t launch_fe3_down(Launch& L, int m, int planes, Tc h, Tc tau, const Tc* E, const typename Cx<Tc>::t* sigma,
                            const typename Cx<Tc>::t* r, typename Cx<Tc>::t* u, typename Cx<Tc>::t* rc) {
  typedef typename Cx<Tc>::t C;
  const double cs = sizeof(C), np = (double)m * m * m * planes;
  const int hm = (m + 1) / 2, mc = (m - 1) / 2;
  cudaError_t e;
  {
    const int cy = fe3_longest(m, 16, fe3_odd_smem<Tc>);
    const size_t odd = fe3_odd_smem<Tc>(m, cy), even = odd / 3;
    if ((e = allow_dynamic_smem(fe3_layer_kernel<Tc, 0>, even)) != cudaSuccess ||
        (e = allow_dynamic_smem(fe3_layer_kernel<Tc, 1>, odd)) != cudaSuccess)
      return e;
    // even rows 0, 2, .., m - 1 in strips of 2 cy rows (the last even row needs no strip of its own)
    const unsigned ns = (unsigned)std::max(1, (mc + cy - 1) / cy);
    const double ev = (double)hm / m, od = (double)mc / m;  // shares of the even and odd layers
    L.begin(KC_MG_SMOOTH);
    fe3_layer_kernel<Tc, 0><<<dim3(ns, (unsigned)hm, (unsigned)planes), kFe3Threads, even, L.stream>>>(r, u, E, sigma,
                                                                                                     m, h, tau, cy);
    if ((e = L.end(KC_MG_SMOOTH, np * ev * 2.0 * cs, np * ev * 100.0)) != cudaSuccess) return e;
    L.begin(KC_MG_SMOOTH);
    fe3_layer_kernel<Tc, 1><<<dim3(ns, (unsigned)mc, (unsigned)planes), kFe3Threads, odd, L.stream>>>(r, u, E, sigma, m,
                                                                                                    h, tau, cy);
    if ((e = L.end(KC_MG_SMOOTH, np * od * 2.0 * cs, np * od * 100.0)) != cudaSuccess) return e;
  }
  const int cy = fe3_longest(m, 8, fe3_restrict_smem<Tc>);
  const size_t smem = fe3_restrict_smem<Tc>(m, cy);
  if ((e = allow_dynamic_smem(fe3_restrict_kernel<Tc>, smem)) != cudaSuccess) return e;
  L.begin(KC_MG_RESID_RESTRICT);
  fe3_restrict_kernel<Tc><<<dim3((unsigned)((mc + cy - 1) / cy), (unsigned)mc, (unsigned)planes), kFe3Threads, smem,
                            L.stream>>>(u, rc, E, sigma, m, h, tau, cy);
  return L.end(KC_MG_RESID_RESTRICT, np * 1.125 * cs, np * 100.0);
}

template <typename Tc>
cudaError_t launch_fe3_tail(Launch& L, int planes, const FeLevels<Tc>& lv, Tc tau, const typename Cx<Tc>::t* sigma,
                            const typename Cx<Tc>::t* r, typename Cx<Tc>::t* u) {
  typedef typename Cx<Tc>::t C;
  size_t n = (size_t)lv.m[0] * lv.m[0] * lv.m[0];
  for (int l = 0; l < lv.count; ++l) n += (size_t)lv.m[l] * lv.m[l] * lv.m[l];
  const size_t smem = n * sizeof(C);
  cudaError_t e = allow_dynamic_smem(fe3_tail_kernel<Tc>, smem);
  if (e != cudaSuccess) return e;
  const double np = (double)lv.m[0] * lv.m[0] * lv.m[0] * planes;
  L.begin(KC_MG_COARSE);
  fe3_tail_kernel<Tc><<<(unsigned)planes, kFe3TailThreads, smem, L.stream>>>(lv, r, u, sigma, tau);
  return L.end(KC_MG_COARSE, 2.0 * np * sizeof(C), 200.0 * np);
}

#define PCOPT_FEMG3(Tc)                                                                                        \
  template bool fe3_down_fits<Tc>(int);                                                                        \
  template cudaError_t launch_fe3_down<Tc>(Launch&, int, int, Tc, Tc, const Tc*, const Cx<Tc>::t*,             \
                                           const Cx<Tc>::t*, Cx<Tc>::t*, Cx<Tc>::t*);                          \
  template cudaError_t launch_fe3_tail<Tc>(Launch&, int, const FeLevels<Tc>&, Tc, const Cx<Tc>::t*,            \
                                           const Cx<Tc>::t*, Cx<Tc>::t*);
PCOPT_FEMG3(float)
PCOPT_FEMG3(double)
#undef PCOPT_FEMG3

}  // namespace pcopt
