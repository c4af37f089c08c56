// In-place shared-memory FFT of many columns, mixed radix 16, 8, 4, 2, 3, 5, 7, used by the
// separable solve of the reduced equations (kern_direct.cu, kern_bottom.cu).
//
// Forward passes are decimation in frequency: pass s splits every span N_s into R parts, transforms
// the R points i + r N_s / R in registers and multiplies output q by exp(-2 pi i q i / N_s). Inputs
// and outputs of a butterfly are the same shared-memory slots, so a pass needs one buffer and one
// barrier; the result stands in digit-reversed order (row perm[k] holds frequency k). The inverse
// runs the passes backwards (twiddle, then butterfly) from that order to the natural one, so no
// reordering pass exists: the real-to-real pre- and post-processing read and write through perm.
// Radix 16 needs two passes for 256 points where radix 4 needs four; the passes through shared
// memory, not the arithmetic, are what bounds the FP32 transforms.
//
// Rows are RP complex values apart, and the R_1 sub-sequences of the first pass start S1 apart
// (S1 = L_1 RP + a pad): consecutive frequencies stand S1 apart, and the pad spreads them over the
// banks for the post-processing.
#pragma once

#include "kern_common.cuh"
#include "snac_impl.h"

namespace snac {
namespace {

template <typename T>
struct alignas(2 * sizeof(T)) Cpl {
  T re, im;
};

template <typename T>
__device__ __forceinline__ Cpl<T> operator+(Cpl<T> a, Cpl<T> b) {
  return {a.re + b.re, a.im + b.im};
}
template <typename T>
__device__ __forceinline__ Cpl<T> operator-(Cpl<T> a, Cpl<T> b) {
  return {a.re - b.re, a.im - b.im};
}
template <typename T>
__device__ __forceinline__ Cpl<T> cx_mul(Cpl<T> a, Cpl<T> b) {
  return {a.re * b.re - a.im * b.im, a.re * b.im + a.im * b.re};
}
// a times conj(b) (inverse twiddles)
template <typename T>
__device__ __forceinline__ Cpl<T> cx_mulc(Cpl<T> a, Cpl<T> b) {
  return {a.re * b.re + a.im * b.im, a.im * b.re - a.re * b.im};
}
// x with its sign flipped if f, on the integer pipe (a selected negation would go to the FP64 pipe)
__device__ __forceinline__ double neg_if(bool f, double x) {
  return __hiloint2double(__double2hiint(x) ^ (f ? (int)0x80000000 : 0), __double2loint(x));
}
__device__ __forceinline__ float neg_if(bool f, float x) { return f ? -x : x; }

// multiplication by -i (forward) or +i (inverse)
template <bool INV, typename T>
__device__ __forceinline__ Cpl<T> rot(Cpl<T> a) {
  return INV ? Cpl<T>{-a.im, a.re} : Cpl<T>{a.im, -a.re};
}

template <bool INV, typename T>
__device__ __forceinline__ void dft4(Cpl<T>& a, Cpl<T>& b, Cpl<T>& c, Cpl<T>& d) {
  const Cpl<T> s = a + c, t = a - c, u = b + d, v = rot<INV>(b - d);
  a = s + u;
  b = t + v;
  c = s - u;
  d = t - v;
}

// In-register DFT of R points (natural order in and out).
template <int R, bool INV, typename T>
__device__ __forceinline__ void dft_reg(Cpl<T> (&x)[R]) {
  if constexpr (R == 2) {
    const Cpl<T> a = x[0], b = x[1];
    x[0] = a + b;
    x[1] = a - b;
  } else if constexpr (R == 4) {
    dft4<INV>(x[0], x[1], x[2], x[3]);
  } else if constexpr (R == 8) {
    // n = 2 n1 + n2: two 4-point DFTs, twiddles exp(-+2 pi i n2 k1 / 8), four 2-point DFTs
    const T h = (T)0.70710678118654752440;
    dft4<INV>(x[0], x[2], x[4], x[6]);
    dft4<INV>(x[1], x[3], x[5], x[7]);
    const T sg = INV ? (T)1 : (T)-1;
    x[3] = Cpl<T>{h * (x[3].re - sg * x[3].im), h * (x[3].im + sg * x[3].re)};
    x[5] = rot<INV>(x[5]);
    x[7] = Cpl<T>{h * (-x[7].re - sg * x[7].im), h * (-x[7].im + sg * x[7].re)};
    // k1 at x[2 k1] (even part) and x[2 k1 + 1] (odd part)
    Cpl<T> y[8];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      y[k] = x[2 * k] + x[2 * k + 1];
      y[k + 4] = x[2 * k] - x[2 * k + 1];
    }
#pragma unroll
    for (int k = 0; k < 8; ++k) x[k] = y[k];
  } else if constexpr (R == 16) {
    // n = 4 n1 + n2: 4-point DFTs over n1, twiddles w16^(n2 k1), 4-point DFTs over n2
    const T c1 = (T)0.92387953251128675613, s1 = (T)0.38268343236508977173, h = (T)0.70710678118654752440;
    const T sg = INV ? (T)1 : (T)-1;
#pragma unroll
    for (int n2 = 0; n2 < 4; ++n2) dft4<INV>(x[n2], x[4 + n2], x[8 + n2], x[12 + n2]);
    // x[4 k1 + n2]
    x[5] = cx_mul(x[5], Cpl<T>{c1, sg * s1});                                                    // w^1
    x[6] = Cpl<T>{h * (x[6].re - sg * x[6].im), h * (x[6].im + sg * x[6].re)};                   // w^2
    x[7] = cx_mul(x[7], Cpl<T>{s1, sg * c1});                                                    // w^3
    x[9] = Cpl<T>{h * (x[9].re - sg * x[9].im), h * (x[9].im + sg * x[9].re)};                   // w^2
    x[10] = rot<INV>(x[10]);                                                                     // w^4
    x[11] = Cpl<T>{h * (-x[11].re - sg * x[11].im), h * (-x[11].im + sg * x[11].re)};            // w^6
    x[13] = cx_mul(x[13], Cpl<T>{s1, sg * c1});                                                  // w^3
    x[14] = Cpl<T>{h * (-x[14].re - sg * x[14].im), h * (-x[14].im + sg * x[14].re)};            // w^6
    x[15] = cx_mul(x[15], Cpl<T>{-c1, -sg * s1});                                                // w^9
#pragma unroll
    for (int k1 = 0; k1 < 4; ++k1) dft4<INV>(x[4 * k1], x[4 * k1 + 1], x[4 * k1 + 2], x[4 * k1 + 3]);
    // X[k1 + 4 k2] stands at x[4 k1 + k2]: transpose
#pragma unroll
    for (int k1 = 0; k1 < 4; ++k1)
#pragma unroll
      for (int k2 = k1 + 1; k2 < 4; ++k2) {
        const Cpl<T> t = x[4 * k1 + k2];
        x[4 * k1 + k2] = x[4 * k2 + k1];
        x[4 * k2 + k1] = t;
      }
  } else {  // 3, 5, 7: pairs p, R - p through their sums and differences
    static_assert(R == 3 || R == 5 || R == 7, "supported radices");
    constexpr int H = (R - 1) / 2;
    constexpr double C3[1] = {-0.5}, S3[1] = {0.86602540378443864676};
    constexpr double C5[2] = {0.30901699437494742410, -0.80901699437494742410};
    constexpr double S5[2] = {0.95105651629515357212, 0.58778525229247312917};
    constexpr double C7[3] = {0.62348980185873353053, -0.22252093395631440429, -0.90096886790241912624};
    constexpr double S7[3] = {0.78183148246802980871, 0.97492791218182360702, 0.43388373911755812048};
    Cpl<T> s[H], d[H];
#pragma unroll
    for (int p = 0; p < H; ++p) {
      s[p] = x[p + 1] + x[R - 1 - p];
      d[p] = x[p + 1] - x[R - 1 - p];
    }
    const Cpl<T> a0 = x[0];
    Cpl<T> sum = a0;
#pragma unroll
    for (int p = 0; p < H; ++p) sum = sum + s[p];
    x[0] = sum;
#pragma unroll
    for (int q = 1; q <= H; ++q) {
      Cpl<T> e = a0, o = {0, 0};  // cosine and sine parts
#pragma unroll
      for (int p = 1; p <= H; ++p) {
        const int m = (p * q) % R;
        const int mm = m <= H ? m : R - m;
        const T c = (T)(R == 3 ? C3[(mm - 1) % 1] : R == 5 ? C5[(mm - 1) % 2] : C7[(mm - 1) % 3]);
        const T sn = (T)((m <= H ? 1.0 : -1.0) * (R == 3 ? S3[(mm - 1) % 1] : R == 5 ? S5[(mm - 1) % 2] : S7[(mm - 1) % 3]));
        e = Cpl<T>{fma(c, s[p - 1].re, e.re), fma(c, s[p - 1].im, e.im)};
        o = Cpl<T>{fma(sn, d[p - 1].re, o.re), fma(sn, d[p - 1].im, o.im)};
      }
      const Cpl<T> ro = rot<INV>(o);  // -i o forward, +i o inverse
      x[q] = e + ro;
      x[R - q] = e - ro;
    }
  }
}

// n / d for 0 <= n < 2^16 - 1 and 1 <= d < 2^16 with r = recip16(d) = floor((2^32 - 1) / d): (n + 1) r / 2^32 is
// less than (n + 1) / d, and by less than 1 / d.
__device__ __forceinline__ int quot16(int n, unsigned r) { return (int)__umulhi((unsigned)n + 1u, r); }

// The columns of a buffer: item t of a pass is (index t / columns, column t % columns).
struct ColsShift {  // 2^lc columns
  int lc;
  __device__ __forceinline__ int cols() const { return 1 << lc; }
  __device__ __forceinline__ int pitch() const { return 1 << lc; }
  __device__ __forceinline__ void split(int t, int& idx, int& c) const {
    idx = t >> lc;
    c = t & ((1 << lc) - 1);
  }
};
struct ColsAny {
  int C, RP;
  unsigned r;  // recip16(C)
  __device__ __forceinline__ int cols() const { return C; }
  __device__ __forceinline__ int pitch() const { return RP; }
  __device__ __forceinline__ void split(int t, int& idx, int& c) const {
    idx = quot16(t, r);
    c = t - idx * C;
  }
};

// Row p of the buffer (p a natural index, or perm[k]).
__device__ __forceinline__ int fft_row(int p, const FftTab& F, int s1, int rp) {
  return quot16(p, F.l1r) * (s1 - F.l1 * rp) + p * rp;
}

template <int R, bool INV, typename T, typename Cols>
__device__ __forceinline__ void fft_pass(Cpl<T>* __restrict__ buf, const FftTab& F, int s, int s1, const Cols cm,
                                         const Cpl<T>* __restrict__ tw, int nt) {
  const int span = F.span[s], L = span / R, tws = F.n / span, rp = cm.pitch();
  const bool first = span == F.n;
  const int stride = first ? s1 : L * rp;
  const int per = first ? 1 : F.l1 / span;
  const int total = (F.n / R) * cm.cols();
  for (int t = threadIdx.x; t < total; t += nt) {
    int idx, c;
    cm.split(t, idx, c);
    int i = idx, o = idx * rp + c;
    if (!first) {
      const int bb = quot16(idx, F.lr[s]);
      i = idx - bb * L;
      const int sub = quot16(bb, F.pr[s]);
      o = sub * s1 + ((bb - sub * per) * span + i) * rp + c;
    }
    Cpl<T> x[R];
#pragma unroll
    for (int r = 0; r < R; ++r) x[r] = buf[o + r * stride];
    if (INV) {
      if (i > 0) {
#pragma unroll
        for (int r = 1; r < R; ++r) x[r] = cx_mulc(x[r], tw[r * i * tws]);
      }
      dft_reg<R, true>(x);
    } else {
      dft_reg<R, false>(x);
      if (i > 0) {
#pragma unroll
        for (int r = 1; r < R; ++r) x[r] = cx_mul(x[r], tw[r * i * tws]);
      }
    }
#pragma unroll
    for (int r = 0; r < R; ++r) buf[o + r * stride] = x[r];
  }
  __syncthreads();
}

// All passes of the forward transform (natural order in, row perm[k] = frequency k out), or of the
// unnormalised inverse. The buffer is complete (behind a barrier) before and after.
template <bool INV, typename T, typename Cols>
__device__ void fft_all(Cpl<T>* __restrict__ buf, const FftTab& F, int s1, const Cols cm, const Cpl<T>* __restrict__ tw,
                        int nt) {
  for (int k = 0; k < F.np; ++k) {
    const int s = INV ? F.np - 1 - k : k;
    switch (F.rad[s]) {
      case 16:
        if constexpr (sizeof(T) == 4) fft_pass<16, INV>(buf, F, s, s1, cm, tw, nt);
        break;
      case 8: fft_pass<8, INV>(buf, F, s, s1, cm, tw, nt); break;
      case 4: fft_pass<4, INV>(buf, F, s, s1, cm, tw, nt); break;
      case 2: fft_pass<2, INV>(buf, F, s, s1, cm, tw, nt); break;
      case 3: fft_pass<3, INV>(buf, F, s, s1, cm, tw, nt); break;
      case 5: fft_pass<5, INV>(buf, F, s, s1, cm, tw, nt); break;
      default: fft_pass<7, INV>(buf, F, s, s1, cm, tw, nt); break;
    }
  }
}

}  // namespace
}  // namespace snac
