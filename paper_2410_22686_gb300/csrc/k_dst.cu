// Sine transforms of grid lines whose m + 1 is not a power of two (or is longer than the
// register FFTs of k_fst.cu): the product with the orthonormal DST-I matrix
// S_ij = sqrt(2/N) sin(pi i j / N), N = m + 1 (Section 2.1, exact spatial solves).
//
// sin(pi i (N - j) / N) = -(-1)^i sin(pi i j / N), so the odd outputs see only the sums
// x_j + x_{N-j} and the even ones only the differences: m^2 / 2 products a line instead of m^2.
// The FP64 kernel is bound by them: 100^2 x 102 planes, an axis pass 344 us with all m^2
// products and 216 with half of them (194 at the FP64 unit's rate), the fused last axis
// 2 x 344 + 35 -> 452.  FP32, bound elsewhere, takes all m products of an output, j ascending:
// a solve preconditioned in FP32 stops where FP32 rounding, amplified by A, stands at rtol, so
// with sums and differences its solution moves by up to rtol (30^2 x 50 at rtol = 1e-8: 1e-8).
// 100^2 x 102 planes in FP32: an axis pass 102 us with one thread a value, 43 from tiles (39
// with half the products), the fused last axis 69 (73).
//
// A CTA of 256 threads holds a tile of lines in shared memory, the line index fastest; a
// thread forms up to four outputs (FP64: of one parity) of its line at a time.  S is read
// through L1, the lines of a tile sharing every value: in FP64 along its columns (S is
// symmetric), in FP32 along its rows.  The last axis of a solve runs fused: transform,
// division by sigma M + tau K on the sine modes, transform.
#include <algorithm>

#include "common.cuh"

namespace pcopt {

namespace {

constexpr int kDstThreads = 256;

// FP64: sums and differences of a line's ends (see the file's head)
template <typename Tc>
constexpr bool dst_folds() {
  return sizeof(Tc) == 8;
}

// Outputs of line c: folded, i = par + 2 (t0 + q G), q < NQ, from the line's sums or
// differences; else i = t0 + q G (par = 0) from the line.
template <typename Tc, int NQ>
__device__ __forceinline__ void dst_outputs(const typename Cx<Tc>::t* src, typename Cx<Tc>::t* dst,
                                            const Tc* __restrict__ S, int m, int lc, int c, int par, int t0, int G) {
  constexpr bool F = dst_folds<Tc>();
  Tc ar[NQ], ai[NQ];
#pragma unroll
  for (int q = 0; q < NQ; ++q) ar[q] = ai[q] = Tc(0);
  const int terms = !F ? m : par == 0 ? (m + 1) / 2 : m / 2;
  // S_ij of output q at s[q * apart]; the next j lies `step` on
  const Tc* s = F ? S + par + 2 * t0 : S + (int64_t)t0 * m;
  const int apart = F ? 2 * G : G * m, step = F ? m : 1;
  for (int j = 0; j < terms; ++j, s += step) {
    const typename Cx<Tc>::t v = src[((par == 0 ? j : m - 1 - j) << lc) + c];
#pragma unroll
    for (int q = 0; q < NQ; ++q) {
      const Tc w = __ldg(s + q * apart);
      ar[q] = fma(w, v.x, ar[q]);
      ai[q] = fma(w, v.y, ai[q]);
    }
  }
#pragma unroll
  for (int q = 0; q < NQ; ++q) {
    const int i = F ? par + 2 * (t0 + q * G) : t0 + q * G;
    dst[(i << lc) + c] = cmk<Tc>(ar[q], ai[q]);
  }
}

// dst = DST-I of every line of src (which ends up as sums and differences where the product
// folds).  Ends with a barrier.
template <typename Tc>
__device__ __forceinline__ void dst_lines(typename Cx<Tc>::t* src, typename Cx<Tc>::t* dst, const Tc* __restrict__ S,
                                          int m, int lc) {
  typedef typename Cx<Tc>::t C;
  constexpr bool F = dst_folds<Tc>();
  const int c = threadIdx.x & ((1 << lc) - 1), g = threadIdx.x >> lc, G = kDstThreads >> lc;
  if (F) {
    for (int j = g; j < m / 2; j += G) {
      const C a = src[(j << lc) + c], b = src[((m - 1 - j) << lc) + c];
      src[(j << lc) + c] = a + b;
      src[((m - 1 - j) << lc) + c] = a - b;
    }
    __syncthreads();
  }
#pragma unroll
  for (int par = 0; par < (F ? 2 : 1); ++par) {
    const int cnt = F ? (m - par + 1) / 2 : m;  // outputs (of this parity)
    for (int t0 = g; t0 < cnt; t0 += 4 * G) {
      switch (min(4, (cnt - t0 + G - 1) / G)) {
        case 4: dst_outputs<Tc, 4>(src, dst, S, m, lc, c, par, t0, G); break;
        case 3: dst_outputs<Tc, 3>(src, dst, S, m, lc, c, par, t0, G); break;
        case 2: dst_outputs<Tc, 2>(src, dst, S, m, lc, c, par, t0, G); break;
        default: dst_outputs<Tc, 1>(src, dst, S, m, lc, c, par, t0, G); break;
      }
    }
  }
  __syncthreads();
}

// Lines along `axis`: plane p = line / (np / m), inside it a line starts at
// outer * m * lstride + inner, lstride = m^axis, inner < lstride.  in may equal out: a CTA
// reads its whole tile before it writes it back.
template <typename Tc, bool DIVIDE>
__global__ void __launch_bounds__(kDstThreads) dst_dense_kernel(const typename Cx<Tc>::t* in, typename Cx<Tc>::t* out,
                                                                const Tc* __restrict__ S, int m, int64_t np,
                                                                int64_t lstride, int64_t nlines, int lc,
                                                                const Tc* __restrict__ lamK,
                                                                const Tc* __restrict__ rmass,
                                                                const typename Cx<Tc>::t* __restrict__ sigma) {
  typedef typename Cx<Tc>::t C;
  extern __shared__ __align__(16) unsigned char dst_smem[];
  C* a = reinterpret_cast<C*>(dst_smem);
  C* b = a + (m << lc);
  __shared__ int64_t lbase[32];  // offset of each line's first value, its plane's included
  __shared__ int lplane[32];     // -1: no line
  const int tid = threadIdx.x, tot = m << lc;
  if (tid < 1 << lc) {
    const int64_t l = ((int64_t)blockIdx.x << lc) + tid, lpp = np / m;
    const int64_t p = l < nlines ? l / lpp : 0, q = l < nlines ? l - p * lpp : 0;
    const int64_t outer = q / lstride;
    lbase[tid] = p * np + outer * lstride * m + (q - outer * lstride);
    lplane[tid] = l < nlines ? (int)p : -1;
  }
  __syncthreads();
  for (int e = tid; e < tot; e += kDstThreads) {
    const int j = e >> lc, c = e & ((1 << lc) - 1);
    a[e] = lplane[c] >= 0 ? in[lbase[c] + (int64_t)j * lstride] : czero<Tc>();
  }
  __syncthreads();
  dst_lines<Tc>(a, b, S, m, lc);
  if (DIVIDE) {
    for (int e = tid; e < tot; e += kDstThreads) {
      const int j = e >> lc, c = e & ((1 << lc) - 1), p = lplane[c];
      if (p < 0) continue;
      const int64_t s = lbase[c] - (int64_t)p * np + (int64_t)j * lstride;  // spectral index in the plane
      C v = b[e];
      if (rmass) v = cscale(v, rmass[s]);  // finite elements: 1 / eigenvalue of M
      b[e] = cmul(v, inv_diag<Tc>(sigma[p], lamK[s]));
    }
    __syncthreads();
    dst_lines<Tc>(b, a, S, m, lc);
  }
  const C* res = DIVIDE ? a : b;
  for (int e = tid; e < tot; e += kDstThreads) {
    const int j = e >> lc, c = e & ((1 << lc) - 1);
    if (lplane[c] >= 0) out[lbase[c] + (int64_t)j * lstride] = res[e];
  }
}

}  // namespace

template <typename Tc>
cudaError_t launch_dst_dense(Launch& L, const Grid& g, int planes, int axis, bool divide, const Tc* S, const Tc* lamK,
                             const Tc* rmass, const typename Cx<Tc>::t* sigma, const typename Cx<Tc>::t* in,
                             typename Cx<Tc>::t* out) {
  typedef typename Cx<Tc>::t C;
  int64_t lstride = 1;
  for (int a = 0; a < axis; ++a) lstride *= g.m;
  const int64_t nlines = (int64_t)planes * (g.np / g.m);
  // lines per CTA: up to 32 in 56 KB (four CTAs an SM), fewer where that leaves less than two
  // CTAs an SM
  auto smem_of = [&](int lc) { return (size_t)2 * sizeof(C) * ((size_t)g.m << lc); };
  int lc = 5;
  while (lc > 0 && (smem_of(lc) > 56 * 1024 || (lc > 1 && (nlines >> lc) < 2 * num_sms()))) --lc;
  const size_t smem = smem_of(lc);
  auto kern = divide ? dst_dense_kernel<Tc, true> : dst_dense_kernel<Tc, false>;
  cudaError_t e = allow_dynamic_smem(kern, smem);
  if (e != cudaSuccess) return e;
  const double tot = (double)planes * (double)g.np;
  const int kc = divide ? KC_FST_DIVIDE : KC_FST_AXIS;
  L.begin(kc);
  kern<<<(unsigned)((nlines + (1 << lc) - 1) >> lc), kDstThreads, smem, L.stream>>>(in, out, S, g.m, g.np, lstride,
                                                                                  nlines, lc, lamK, rmass, sigma);
  return L.end(kc, 2.0 * tot * sizeof(C), (divide ? 2.0 : 1.0) * tot * (dst_folds<Tc>() ? 2.0 : 4.0) * g.m);
}

template cudaError_t launch_dst_dense<float>(Launch&, const Grid&, int, int, bool, const float*, const float*,
                                             const float*, const float2*, const float2*, float2*);
template cudaError_t launch_dst_dense<double>(Launch&, const Grid&, int, int, bool, const double*, const double*,
                                              const double*, const double2*, const double2*, double2*);

}  // namespace pcopt
