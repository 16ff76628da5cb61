// Scaled FFT along time for lengths that are not powers of two (the paper's own runs
// use n = 2^k - 1): the same two-for-one transform as k_tfft.cu by Bluestein's chirp-z
// method (L. I. Bluestein, IEEE Trans. Audio Electroacoust. 18, 1970).  With
// j k = (j^2 + k^2 - (k - j)^2) / 2 and c_j = exp(-pi i j^2 / n),
//   X_k = c_k sum_j (x_j c_j) conj(c_{k-j}),
// a convolution with the chirp, taken cyclically in M = 2^b >= 2n points.
//
// A CTA holds COLS spatial columns of M complex values in shared memory.  The forward
// M-point transform is a decimation in frequency by register DFTs of 8 or 16 points and
// the inverse its mirror image (decimation in time), so neither reorders: the chirp's
// spectrum is stored in the digit-reversed order the forward passes leave, and the last
// forward pass, the product with it and the first inverse pass stay in registers.  The
// first pass knows that its upper half is zero and the last one forms the lower half only.
//
// The FP64 unit bounds the FP64 transforms: the direct sum takes 8 (n/2 + 1) n operations a
// column, this about 66 M (n = 511: 1.05 M against 68 k; 63^2 columns: 8.17 -> 0.6 ms a
// transform).  The direct sum of k_tfft.cu stays below n = 24, where its rounding error is
// the smaller one (n = 20, FP64: 1.31e-15 against 1.49e-15; from 24 on this one's is no
// larger, n = 511 in FP32: 3.0e-6 against 1.4e-6).  31^2 columns, forward, FP64: n = 24
// 53.5 -> 17.2 us, n = 31 71.9 -> 16.8, n = 100 343 -> 39, n = 511 2058 -> 162;
// FP32: n = 24 12.6 -> 7.8, n = 100 77.9 -> 10.6, n = 511 391 -> 19.
//
// FP32 transforms around sine-transform solves and BF16 storage keep the direct sum at every
// length: what such a solve leaves at rtol is FP32 rounding amplified by A (or flipped BF16
// roundings), and another order of the sums moves its solution by up to rtol (31^2 x 63 at rtol =
// 1e-8: 9.5e-9).  Around multigrid with FP32 storage the cycle's own error is what is left
// there, and the solutions agree to 1e-12.
#include <algorithm>

#include "common.cuh"
#include "finecorr.cuh"
#include "regfft.cuh"

namespace pcopt {

namespace {

constexpr int kCzThreads = 256;

// log2 of the radix of the next pass when `rem` bits of the length are left (rem >= 3)
__host__ __device__ __forceinline__ int cz_bits(int rem) { return rem == 3 || rem == 6 || rem == 9 ? 3 : 4; }

// sm is [M][COLS], COLS = 1 << lc; filt and roots as in ChirpZ
template <typename Tc>
struct CzTile {
  typename Cx<Tc>::t* sm;
  const typename Cx<Tc>::t* roots;
  int M, lc;
};

// one forward pass over sub-transforms of length L = R S: R-point DFTs of the elements S
// apart, times w_L^{p r}.  FIRST: elements n.. (and so the upper half) are zero.
template <typename Tc, int R, bool FIRST>
__device__ __forceinline__ void cz_forward_pass(const CzTile<Tc>& t, int lS, int n) {
  typedef typename Cx<Tc>::t C;
  const int S = 1 << lS, step = t.M / (R * S);
  const int tasks = (t.M / R) << t.lc;
  for (int e = threadIdx.x; e < tasks; e += kCzThreads) {
    const int c = e & ((1 << t.lc) - 1), g = e >> t.lc;
    const int p = g & (S - 1);
    const int base = (g - p) * R + p;
    C x[R];
#pragma unroll
    for (int q = 0; q < R; ++q) {
      if (FIRST && q >= R / 2) {
        x[q] = czero<Tc>();
      } else {
        const int i = base + q * S;
        x[q] = !FIRST || i < n ? t.sm[(i << t.lc) + c] : czero<Tc>();
      }
    }
    dft_regs<R, false, FIRST>(x);
#pragma unroll
    for (int r = 0; r < R; ++r)
      t.sm[((base + r * S) << t.lc) + c] = r == 0 ? x[0] : cmul(t.roots[p * r * step], x[r]);
  }
  __syncthreads();
}

// the last forward pass (S = 1), the product with the chirp's spectrum, the first inverse pass
template <typename Tc, int R>
__device__ __forceinline__ void cz_middle_pass(const CzTile<Tc>& t, const typename Cx<Tc>::t* __restrict__ filt) {
  typedef typename Cx<Tc>::t C;
  const int tasks = (t.M / R) << t.lc;
  for (int e = threadIdx.x; e < tasks; e += kCzThreads) {
    const int c = e & ((1 << t.lc) - 1), base = (e >> t.lc) * R;
    C x[R];
#pragma unroll
    for (int q = 0; q < R; ++q) x[q] = t.sm[((base + q) << t.lc) + c];
    dft_regs<R, false>(x);
#pragma unroll
    for (int q = 0; q < R; ++q) x[q] = cmul(filt[base + q], x[q]);
    dft_regs<R, true>(x);
#pragma unroll
    for (int q = 0; q < R; ++q) t.sm[((base + q) << t.lc) + c] = x[q];
  }
  __syncthreads();
}

// one inverse pass; LAST: outputs k < n only, times the chirp
template <typename Tc, int R, bool LAST>
__device__ __forceinline__ void cz_inverse_pass(const CzTile<Tc>& t, int lS, int n,
                                                const typename Cx<Tc>::t* __restrict__ chirp) {
  typedef typename Cx<Tc>::t C;
  const int S = 1 << lS, step = t.M / (R * S);
  const int tasks = (t.M / R) << t.lc;
  for (int e = threadIdx.x; e < tasks; e += kCzThreads) {
    const int c = e & ((1 << t.lc) - 1), g = e >> t.lc;
    const int p = g & (S - 1);
    const int base = (g - p) * R + p;
    C x[R];
#pragma unroll
    for (int r = 0; r < R; ++r) {
      x[r] = t.sm[((base + r * S) << t.lc) + c];
      if (r != 0) x[r] = cmul(cconj(t.roots[p * r * step]), x[r]);
    }
    dft_regs<R, true, false, LAST>(x);
#pragma unroll
    for (int q = 0; q < (LAST ? R / 2 : R); ++q) {
      const int i = base + q * S;
      if (!LAST)
        t.sm[(i << t.lc) + c] = x[q];
      else if (i < n)
        t.sm[(i << t.lc) + c] = cmul(chirp[i], x[q]);
    }
  }
  __syncthreads();
}

// the n-point DFT of sm[0..n-1] (already times the chirp) in place
template <typename Tc>
__device__ __forceinline__ void cz_transform(const CzTile<Tc>& t, int logM, int n,
                                             const typename Cx<Tc>::t* __restrict__ chirp,
                                             const typename Cx<Tc>::t* __restrict__ filt) {
  // radices: bits b0, b1, .. from the top; M >= 64, so there are at least two passes
  int rem = logM - cz_bits(logM);
  if (cz_bits(logM) == 4)
    cz_forward_pass<Tc, 16, true>(t, rem, n);
  else
    cz_forward_pass<Tc, 8, true>(t, rem, n);
  while (rem > 4) {
    const int b = cz_bits(rem);
    rem -= b;
    if (b == 4)
      cz_forward_pass<Tc, 16, false>(t, rem, n);
    else
      cz_forward_pass<Tc, 8, false>(t, rem, n);
  }
  if (rem == 4)
    cz_middle_pass<Tc, 16>(t, filt);
  else
    cz_middle_pass<Tc, 8>(t, filt);
  // the same passes from the shortest sub-transform up
  int done = rem;
  while (true) {
    // the pass whose sub-transforms have length 2^(done + b): the forward radices in reverse
    int r = logM, b = 0;
    while (r > done) {
      b = cz_bits(r);
      r -= b;
    }
    if (done + b == logM) {
      if (b == 4)
        cz_inverse_pass<Tc, 16, true>(t, done, n, chirp);
      else
        cz_inverse_pass<Tc, 8, true>(t, done, n, chirp);
      return;
    }
    if (b == 4)
      cz_inverse_pass<Tc, 16, false>(t, done, n, chirp);
    else
      cz_inverse_pass<Tc, 8, false>(t, done, n, chirp);
    done += b;
  }
}

template <typename Tc, typename Tin>
__global__ void __launch_bounds__(kCzThreads, 2) tchirp_forward_kernel(const Tin* __restrict__ v,
                                                                       const Tc* __restrict__ dpow,
                                                                       ChirpZ<Tc> cz,
                                                                       typename Cx<Tc>::t* __restrict__ spec,
                                                                       int64_t ms, int n, int lc) {
  typedef typename Cx<Tc>::t C;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const CzTile<Tc> t{reinterpret_cast<C*>(smem_raw), cz.roots(n), 1 << cz.logM, lc};
  const int64_t s0 = (int64_t)blockIdx.x << lc;
  const Tin* v1 = v;
  const Tin* v2 = v + (int64_t)n * ms;
  for (int e = threadIdx.x; e < n << lc; e += kCzThreads) {
    const int j = e >> lc;
    const int64_t s = s0 + (e & ((1 << lc) - 1));
    C z = czero<Tc>();
    if (s < ms) {
      const Tc d = dpow[j];
      z = cmk<Tc>(cvt<Tc>(v1[(int64_t)(n - 1 - j) * ms + s]) * d, cvt<Tc>(v2[(int64_t)j * ms + s]) * d);
    }
    t.sm[e] = cmul(cz.chirp()[j], z);  // D J v1 + i D v2
  }
  __syncthreads();
  cz_transform<Tc>(t, cz.logM, n, cz.chirp(), cz.filter(n));
  const int nf = n / 2 + 1;
  for (int e = threadIdx.x; e < nf << lc; e += kCzThreads) {
    const int k = e >> lc, c = e & ((1 << lc) - 1);
    const int64_t s = s0 + c;
    if (s >= ms) continue;
    const C Z = t.sm[(k << lc) + c];
    const C W = t.sm[((k == 0 ? 0 : n - k) << lc) + c];
    // 2 hat v2[k] = -i (Z[k] - conj Z[n-k]);  2 hat v1[k] = Z[k] + conj Z[n-k] (as k_tfft.cu)
    spec[(int64_t)(2 * k) * ms + s] = cmk<Tc>(Z.y + W.y, W.x - Z.x);
    spec[(int64_t)(2 * k + 1) * ms + s] = cmk<Tc>(Z.x + W.x, Z.y - W.y);
  }
}

// The inverse transform is the forward one with real and imaginary parts exchanged on
// both sides.
template <typename Tc, typename Tout>
__global__ void __launch_bounds__(kCzThreads, 2) tchirp_inverse_kernel(const typename Cx<Tc>::t* __restrict__ spec,
                                                                       const Tc* __restrict__ dinv, ChirpZ<Tc> cz,
                                                                       Tout* __restrict__ w, int64_t ms, int n, int lc,
                                                                       FineCorrection<typename Cx<Tc>::t> fc) {
  typedef typename Cx<Tc>::t C;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const CzTile<Tc> t{reinterpret_cast<C*>(smem_raw), cz.roots(n), 1 << cz.logM, lc};
  const int64_t s0 = (int64_t)blockIdx.x << lc;
  const int nf = n / 2 + 1;
  for (int e = threadIdx.x; e < nf << lc; e += kCzThreads) {
    const int k = e >> lc, c = e & ((1 << lc) - 1);
    const int64_t s = s0 + c;
    C sa = czero<Tc>(), sb = czero<Tc>();
    if (s < ms) {
      sa = spec[(int64_t)(2 * k) * ms + s];
      sb = spec[(int64_t)(2 * k + 1) * ms + s];
      if (fc.ec) {
        Parents<Tc, C> par;
        par.init(fc, s);
        sa = par.corrected(sa, fc, 2 * k);
        sb = par.corrected(sb, fc, 2 * k + 1);
      }
    }
    // Y[k] = hat w1[k] + i hat w2[k], Y[n-k] = conj(hat w1[k]) + i conj(hat w2[k]), exchanged
    t.sm[(k << lc) + c] = cmul(cz.chirp()[k], cmk<Tc>(sb.y + sa.x, sb.x - sa.y));
    if (k > 0 && 2 * k < n) t.sm[((n - k) << lc) + c] = cmul(cz.chirp()[n - k], cmk<Tc>(sa.x - sb.y, sb.x + sa.y));
  }
  __syncthreads();
  cz_transform<Tc>(t, cz.logM, n, cz.chirp(), cz.filter(n));
  Tout* w1 = w;
  Tout* w2 = w + (int64_t)n * ms;
  for (int e = threadIdx.x; e < n << lc; e += kCzThreads) {
    const int j = e >> lc, c = e & ((1 << lc) - 1);
    const int64_t s = s0 + c;
    if (s >= ms) continue;
    const int jr = n - 1 - j;
    const Tc wt1 = dinv[jr] * t.sm[(jr << lc) + c].y;  // J D^{-1} ifft(hat w1)
    const Tc wt2 = dinv[j] * t.sm[(j << lc) + c].x;    // D^{-1} ifft(hat w2)
    w1[(int64_t)j * ms + s] = cvt<Tout>(wt1 - wt2);  // step 4: [[I, -I], [I, I]]
    w2[(int64_t)j * ms + s] = cvt<Tout>(wt1 + wt2);
  }
}

// log2 of the columns a CTA holds: 64 KB of shared memory (two to three CTAs an SM), at
// most 64 columns, at least one (M = 8192 in FP64: 128 KB), and fewer (to a 32-byte
// sector of the vector's rows) where that leaves fewer than two CTAs an SM
template <typename Tc>
int cz_lc(int logM, int64_t ms) {
  const int room = sizeof(Tc) == 8 ? 12 : 13, least = sizeof(Tc) == 8 ? 2 : 3;
  int lc = std::max(0, std::min(6, room - logM));
  while (lc > least && (ms >> lc) < 2 * num_sms()) --lc;
  return lc;
}

}  // namespace

int chirp_log2(int n) {
  if (n < kChirpMinN || (n & (n - 1)) == 0) return 0;
  int b = 1;
  while ((1 << b) < 2 * n) ++b;
  return b;
}

int chirp_position(int logM, int k) {
  int pos = 0;
  for (int rem = logM; rem > 0;) {
    const int b = cz_bits(rem);
    rem -= b;
    pos += (k & ((1 << b) - 1)) << rem;
    k >>= b;
  }
  return pos;
}

template <typename Tc, typename Tin>
cudaError_t launch_tchirp_forward(Launch& L, int64_t ms, int n, const Tin* v, const Tc* dpow, ChirpZ<Tc> cz,
                                  typename Cx<Tc>::t* spec) {
  typedef typename Cx<Tc>::t C;
  const int lc = cz_lc<Tc>(cz.logM, ms);
  const size_t smem = sizeof(C) << (cz.logM + lc);
  auto kern = tchirp_forward_kernel<Tc, Tin>;
  cudaError_t e = allow_dynamic_smem(kern, smem);
  if (e != cudaSuccess) return e;
  L.begin(KC_TFFT_FWD);
  kern<<<(unsigned)((ms + (1 << lc) - 1) >> lc), kCzThreads, smem, L.stream>>>(v, dpow, cz, spec, ms, n, lc);
  return L.end(KC_TFFT_FWD, 2.0 * n * ms * sizeof(Tin) + 2.0 * (n / 2 + 1) * ms * sizeof(C),
               (double)ms * (10.0 * cz.logM + 6.0) * (1 << cz.logM));
}

template <typename Tc, typename Tout>
cudaError_t launch_tchirp_inverse(Launch& L, int64_t ms, int n, const typename Cx<Tc>::t* spec, const Tc* dinv,
                                  ChirpZ<Tc> cz, Tout* w, FineCorrection<typename Cx<Tc>::t> fc) {
  typedef typename Cx<Tc>::t C;
  const int lc = cz_lc<Tc>(cz.logM, ms);
  const size_t smem = sizeof(C) << (cz.logM + lc);
  auto kern = tchirp_inverse_kernel<Tc, Tout>;
  cudaError_t e = allow_dynamic_smem(kern, smem);
  if (e != cudaSuccess) return e;
  const double cbytes = fc.ec ? (double)(n / 2 + 1) * 2.0 * fc.npc * sizeof(C) : 0.0;
  L.begin(KC_TFFT_INV);
  kern<<<(unsigned)((ms + (1 << lc) - 1) >> lc), kCzThreads, smem, L.stream>>>(spec, dinv, cz, w, ms, n, lc, fc);
  return L.end(KC_TFFT_INV, 2.0 * (n / 2 + 1) * ms * sizeof(C) + 2.0 * n * ms * sizeof(Tout) + cbytes,
               (double)ms * (10.0 * cz.logM + 6.0) * (1 << cz.logM));
}

template cudaError_t launch_tchirp_forward<double, double>(Launch&, int64_t, int, const double*, const double*,
                                                           ChirpZ<double>, double2*);
template cudaError_t launch_tchirp_forward<float, double>(Launch&, int64_t, int, const double*, const float*,
                                                          ChirpZ<float>, float2*);
template cudaError_t launch_tchirp_forward<float, float>(Launch&, int64_t, int, const float*, const float*,
                                                         ChirpZ<float>, float2*);
#define PCOPT_INV(Tc, Tout)                                                                                       \
  template cudaError_t launch_tchirp_inverse<Tc, Tout>(Launch&, int64_t, int, const Cx<Tc>::t*, const Tc*, ChirpZ<Tc>, \
                                                       Tout*, FineCorrection<Cx<Tc>::t>);
PCOPT_INV(double, double)
PCOPT_INV(float, double)
PCOPT_INV(float, float)
#undef PCOPT_INV

}  // namespace pcopt
