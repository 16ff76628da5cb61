// Radix-2 FFT of a small power-of-two length held in registers (one thread
// owns the whole sequence) and the cp.async helpers, shared by the time FFTs and
// the sine transforms.
#pragma once

#include "common.cuh"

namespace pcopt {

template <int R>
__device__ __forceinline__ constexpr int brev_ct(int i) {
  int r = 0;
  for (int b = 1, rb = R >> 1; b < R; b <<= 1, rb >>= 1)
    if (i & b) r |= rb;
  return r;
}

// cos(2 pi q / 32) for q = 0..8; q = 8 as the FP64 cosine of the rounded pi / 2 (what the
// host-made twiddle tables hold)
template <typename T>
__device__ __forceinline__ constexpr T cos32(int q) {
  switch (q) {
    case 0: return T(1);
    case 1: return T(0.98078528040323044912618223613424);
    case 2: return T(0.92387953251128675612818318939679);
    case 3: return T(0.83146961230254523707878837761791);
    case 4: return T(0.70710678118654752440084436210485);
    case 5: return T(0.55557023301960222474283081394853);
    case 6: return T(0.38268343236508977172845998403040);
    case 7: return T(0.19509032201612826784828486847702);
    default: return T(6.123233995736766e-17);
  }
}

// In-place R-point DFT of registers (R <= 32), the twiddles compile-time constants.  In FP64,
// whose unit bounds the transforms, quarter turns cost their two sums alone and a butterfly
// with another twiddle takes six fused multiply-adds (a + w b in four, a - w b as
// 2 a - (a + w b)) where a product and two sums take eight: 148 operations for 16 points
// instead of 196 (preconditioner apply in FP64, 31^2: n = 256 2.24e-15 off against 2.26e-15
// before).  In FP32, bound elsewhere, every twiddle is a product followed by the sums, quarter
// turns too (their cosine is 6e-17): the values of the twiddle tables, bit for bit.  A solve
// preconditioned in FP32 stops where FP32 rounding, amplified by A, stands at rtol, so another
// order of these operations moves its solution by up to rtol (at rtol = 1e-8, 63^2 x 64, by
// 4e-9).  HALF_IN: inputs R/2.. are zero; HALF_OUT: only outputs 0..R/2-1 are wanted.
template <int R, bool INV, bool HALF_IN = false, bool HALF_OUT = false, typename C>
__device__ __forceinline__ void dft_regs(C (&x)[R]) {
  typedef decltype(C().x) T;
#pragma unroll
  for (int i = 0; i < R; ++i) {
    const int j = brev_ct<R>(i);
    if (j > i) {
      const C t = x[i];
      x[i] = x[j];
      x[j] = t;
    }
  }
#pragma unroll
  for (int half = 1; half < R; half <<= 1) {
    const bool last = HALF_OUT && 2 * half == R;
#pragma unroll
    for (int g = 0; g < R; g += 2 * half) {
#pragma unroll
      for (int p = 0; p < half; ++p) {
        const C a = x[g + p], b = x[g + p + half];
        if (HALF_IN && half == 1) {
          x[g + 1] = a;
        } else if (p == 0) {
          x[g + p] = a + b;
          if (!last) x[g + p + half] = a - b;
        } else if (sizeof(T) == 8 && 2 * p == half) {  // w = -i (forward), i (inverse)
          C t;
          t.x = INV ? -b.y : b.y;
          t.y = INV ? b.x : -b.x;
          x[g + p] = a + t;
          if (!last) x[g + p + half] = a - t;
        } else {
          const int q = p * (16 / half);  // w = exp(-+ 2 pi i q / 32), 0 < q < 16
          const T wr = q <= 8 ? cos32<T>(q) : -cos32<T>(16 - q);
          const T ws = q <= 8 ? cos32<T>(8 - q) : cos32<T>(q - 8);
          const T wi = INV ? ws : -ws;
          C t;
          if (sizeof(T) == 8) {
            t.x = fma(-wi, b.y, fma(wr, b.x, a.x));
            t.y = fma(wi, b.x, fma(wr, b.y, a.y));
            x[g + p] = t;
            if (!last) {
              x[g + p + half].x = fma(T(2), a.x, -t.x);
              x[g + p + half].y = fma(T(2), a.y, -t.y);
            }
          } else {
            // rounded as the product with a twiddle from memory: constants may be contracted otherwise
            t.x = fma(wr, b.x, -__fmul_rn(wi, b.y));
            t.y = fma(wr, b.y, __fmul_rn(wi, b.x));
            x[g + p] = a + t;
            if (!last) x[g + p + half] = a - t;
          }
        }
      }
    }
  }
}

// cp.async (sm_80+ asynchronous global -> shared copy of B = 4, 8 or 16 bytes,
// bypassing registers); `ok == false` zero-fills the destination without reading
// global memory
template <int B>
__device__ __forceinline__ void cp_async(void* dst, const void* src, bool ok) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
  const int sz = ok ? B : 0;
  asm volatile("cp.async.ca.shared.global [%0], [%1], %2, %3;\n" ::"r"(d), "l"(src), "n"(B), "r"(sz) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory");
}

}  // namespace pcopt
