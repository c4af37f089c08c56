// Transforms along the homogeneous direction (Table 1) for lengths whose half has no prime factor above
// 7: one chunk of C = 2^lc columns per CTA on the in-place FFT of fft_dev.cuh. Each column is its own
// half-length complex sequence (conventions and reductions as listed in kern_transform.cu), so columns
// of very different magnitude do not meet. Compared with the Stockham stages of transform_dev.cuh (which
// keep the other lengths): one buffer instead of two, half as many passes through shared memory
// (radix 16 / 8), and the real-DFT split done once per pair of bins (one twiddle product for four
// outputs: 16 FP64 operations per value at n = 256 in place of 21; sign flips on the integer pipe). The FP64
// kernels are bound by the FP64 pipe (85 % active), the FP32 ones by instruction issue and the latency of
// the strided loads. Measured forward / backward, before -> now: 512 x 512 x 256 FP32 0.34 -> 0.24 / 0.45 ->
// 0.30 ms, FP64 2.65 -> 2.15 / 2.35 -> 2.28 ms; 20011 columns of 576 FP64 0.73 -> 0.50 / 0.67 -> 0.51 ms.
#pragma once

#include "fft_dev.cuh"
#include "transform_dev.cuh"

namespace snac {
namespace {

template <typename T>
struct ZArgs {
  FftTab F;  // length m = n / 2
  int n, kind, lc;
  const Cpl<T>* fft;   // e^{-2 pi i k / m}
  const Cpl<T>* twn;   // e^{-2 pi i k / n}, k = 0..m
  const Cpl<T>* tw2n;  // e^{-i pi k / 2n}, k = 0..n
  const Cpl<T>* tw4a;  // e^{-i pi (4k+1) / 4n}
  const Cpl<T>* tw4b;  // e^{-i pi k / n}
  const int* perm;     // row of frequency k
};

template <typename T>
inline ZArgs<T> z_args(const snac_plan* P, int tc) {
  ZArgs<T> A{};
  const Cpl<T>* t = reinterpret_cast<const Cpl<T>*>(sizeof(T) == 8 ? (const void*)P->d_tw64 : (const void*)P->d_tw32);
  A.F = P->zfft;
  A.n = P->nzt;
  A.kind = P->kind;
  while ((1 << A.lc) < tc) ++A.lc;
  A.fft = t + P->tw.fft;
  A.twn = t + P->tw.twn;
  A.tw2n = t + P->tw.tw2n;
  A.tw4a = t + P->tw.tw4a;
  A.tw4b = t + P->tw.tw4b;
  A.perm = P->d_zperm;
  return A;
}

// Caller offsets (at k = 0) of the chunk's columns and the caller stride along the homogeneous axis.
__device__ __forceinline__ long long z_columns(const ChunkDev& ch, const BlockDev& B, const CallerBlk* __restrict__ cb,
                                               int cols, long long* coff) {
  const CallerBlk C = cb[ch.b];
  if ((int)threadIdx.x < cols) {
    const int pc = ch.c0 + threadIdx.x;
    coff[threadIdx.x] = C.off3 + (long long)(pc % B.nx) * C.s[0] + (long long)(pc / B.nx) * C.s[1];
  }
  __syncthreads();
  return C.s[2];
}

constexpr int ZMAXC = 64;
constexpr int ZLB = 8;  // column loads in flight per thread

// Forward transform of one chunk by a CTA of nt threads: in3 (caller layout) -> out [q][cell].
template <typename T, typename TI>
__device__ void z_forward(const ZArgs<T>& A, const ChunkDev ch, const BlockDev* __restrict__ blk,
                          const CallerBlk* __restrict__ cb, const TI* __restrict__ in3, T* __restrict__ out,
                          long long ncell, T sub0, int split, unsigned char* smem, int nt) {
  __shared__ long long coff[ZMAXC];
  __shared__ long long ooff[ZMAXC];
  const int lc = A.lc, C = 1 << lc, n = A.n, m = n / 2, kind = A.kind;
  Cpl<T>* buf = reinterpret_cast<Cpl<T>*>(smem);
  T* bt = reinterpret_cast<T*>(smem);
  const BlockDev B = blk[ch.b];
  if ((int)threadIdx.x < C) {
    const int pc = ch.c0 + threadIdx.x;
    ooff[threadIdx.x] = split ? split_cell(B, pc % B.nx, pc / B.nx) : B.off + pc;
  }
  const long long sk = z_columns(ch, B, cb, C, coff);  // (its barrier also covers ooff)
  const bool flip = kind == KIND_DD || kind == KIND_DN, four = kind == KIND_ND || kind == KIND_DN;
  const int c = threadIdx.x & (C - 1), r0 = threadIdx.x >> lc, rs = nt >> lc;
  const bool live = c < ch.ncol;
  // cell k of column cc goes to component t & 1 of row t / 2 (four: row and component of t_j)
  auto put = [&](int k, int cc, TI v) {
    const T x = neg_if(flip && (k & 1), to_inner<T, TI>(v));
    int o;
    if (four) o = ((((k & 1) ? (n - 1 - k) >> 1 : k >> 1) << lc) + cc) * 2 + (k & 1);
    else {
      const int t = kind == KIND_PP ? k : ((k & 1) ? n - 1 - (k >> 1) : (k >> 1));
      o = (((t >> 1) << lc) + cc) * 2 + (t & 1);
    }
    bt[o] = x;
  };
  if (sk != 1) {  // a row of the chunk is C consecutive cells; column c is this thread's
    const TI* src = in3 + (live ? coff[c] : 0);
    for (int k0 = r0; k0 < n; k0 += ZLB * rs) {
      TI v[ZLB];
#pragma unroll
      for (int u = 0; u < ZLB; ++u) {
        const int k = k0 + u * rs;
        v[u] = live && k < n ? src[(long long)k * sk] : (TI)0;
      }
#pragma unroll
      for (int u = 0; u < ZLB; ++u) {
        const int k = k0 + u * rs;
        if (k < n) put(k, c, v[u]);
      }
    }
  } else {  // the homogeneous axis is the caller's contiguous one: consecutive threads run along it
    for (int i = threadIdx.x; i < n << lc; i += nt) {
      const int cc = i / n, k = i - cc * n;
      put(k, cc, cc < ch.ncol ? in3[coff[cc] + k] : (TI)0);
    }
  }
  __syncthreads();
  const ColsShift cm{lc};
  if (four) {
    for (int j = r0; j < m; j += rs) buf[(j << lc) + c] = cx_mul(buf[(j << lc) + c], A.tw4a[j]);
    __syncthreads();
  }
  fft_all<false>(buf, A.F, A.F.l1 << lc, cm, A.fft, nt);
  T* ob = out + (live ? ooff[c] : 0);
  auto store = [&](int q, T y) {
    if (live) ob[(long long)q * ncell] = y;
  };
  if (four) {
    for (int k = r0; k < m; k += rs) {
      const Cpl<T> v = cx_mul(buf[(A.perm[k] << lc) + c], A.tw4b[k]);
      const int q = 2 * k;
      store(kind == KIND_DN ? n - 1 - q : q, (T)2 * v.re);
      store(kind == KIND_DN ? q : n - 1 - q, (T)-2 * v.im);
    }
    return;
  }
  // twice the spectrum X of the length-n real sequence at bin b: outputs b and n - b
  auto emit = [&](int b, Cpl<T> x) {
    const bool mirror = b > 0 && b < m;
    if (kind == KIND_PP) {
      store(b, (T)0.5 * x.re);
      if (mirror) store(n - b, (T)0.5 * x.im);
    } else {
      const Cpl<T> w = A.tw2n[b];
      store(kind == KIND_DD ? n - 1 - b : b, w.re * x.re - w.im * x.im);
      if (mirror) store(kind == KIND_DD ? b - 1 : n - b, -w.im * x.re - w.re * x.im);
    }
  };
  for (int k = r0; k <= m / 2; k += rs) {
    const Cpl<T> a = buf[(A.perm[k] << lc) + c];
    const Cpl<T> b = k == 0 ? a : buf[(A.perm[m - k] << lc) + c];
    const Cpl<T> e = {a.re + b.re, a.im - b.im};
    const Cpl<T> o = cx_mul(Cpl<T>{a.im + b.im, b.re - a.re}, A.twn[k]);  // w^k times -i (a - conj b)
    emit(k, e + o);
    if (m - k != k) emit(m - k, Cpl<T>{e.re - o.re, o.im - e.im});  // conj(e - o)
  }
  // F(x - shift0) = F(x) - shift0 F(1), which is zero outside mode 0 (this thread's own output)
  if (sub0 != (T)0 && r0 == 0 && live) ob[0] -= sub0;
}

// Inverse transform of one chunk and update: p3 += inv_theta F^-1 of modes.
template <typename T>
__device__ void z_backward(const ZArgs<T>& A, const ChunkDev ch, const BlockDev* __restrict__ blk,
                           const CallerBlk* __restrict__ cb, const T* __restrict__ modes, double* __restrict__ p3,
                           long long ncell, double inv_theta, unsigned char* smem, int nt) {
  __shared__ long long coff[ZMAXC];
  const int lc = A.lc, C = 1 << lc, n = A.n, m = n / 2, kind = A.kind;
  Cpl<T>* buf = reinterpret_cast<Cpl<T>*>(smem);
  const BlockDev B = blk[ch.b];
  const long long sk = z_columns(ch, B, cb, C, coff);
  const bool flip = kind == KIND_DD || kind == KIND_DN, four = kind == KIND_ND || kind == KIND_DN;
  const int c = threadIdx.x & (C - 1), r0 = threadIdx.x >> lc, rs = nt >> lc;
  const bool live = c < ch.ncol;
  if (sk != 1 && threadIdx.x < 32) {
    // p is read only after the transform: bring its rows to L2 meanwhile (one 128-byte line per row,
    // two where the chunk straddles a line)
    for (int j = threadIdx.x; j < n; j += 32) {
      const double* a = p3 + (long long)j * sk;
      asm volatile("prefetch.global.L2 [%0];" ::"l"(a + coff[0]));
      asm volatile("prefetch.global.L2 [%0];" ::"l"(a + coff[ch.ncol - 1]));
    }
  }
  const T* src = modes + B.off + ch.c0 + (live ? c : 0);
  auto X = [&](int q) -> T {  // coefficient q of the DCT (the DST kinds store theirs reversed); 0 past the end
    if (!live || q >= n) return (T)0;
    return src[(long long)(flip ? n - 1 - q : q) * ncell];
  };
  if (four) {
    for (int j0 = r0; j0 < m; j0 += 4 * rs) {
      T a[4], b[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int j = j0 + u * rs;
        a[u] = j < m ? X(2 * j) : (T)0;
        b[u] = j < m ? X(n - 1 - 2 * j) : (T)0;
      }
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int j = j0 + u * rs;
        if (j >= m) continue;
        const Cpl<T> v = cx_mul(Cpl<T>{a[u], b[u]}, A.tw4a[j]);
        buf[(A.perm[j] << lc) + c] = Cpl<T>{v.re, -v.im};  // forward = conj(inverse(conj))
      }
    }
  } else {
    for (int k0 = r0; k0 <= m / 2; k0 += 2 * rs) {
      T x[2][4];
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        const int k = k0 + u * rs;
        const bool in = k <= m / 2;
        x[u][0] = in ? X(k) : (T)0;
        x[u][1] = in && k > 0 ? X(n - k) : (T)0;
        x[u][2] = in ? X(m - k) : (T)0;
        x[u][3] = in ? X(m + k) : (T)0;
      }
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        const int k = k0 + u * rs;
        if (k > m / 2) continue;
        // half-spectrum bins k and m - k: PP the stored (X_b, X_{n-b}); NN/DD e^{+i pi b/2n} (X_b - i X_{n-b})
        Cpl<T> b1, b2;
        if (kind == KIND_PP) {
          b1 = Cpl<T>{x[u][0], x[u][1]};
          b2 = Cpl<T>{x[u][2], k == 0 ? (T)0 : x[u][3]};
        } else {
          const Cpl<T> w = A.tw2n[k], v = A.tw2n[m - k];
          b1 = cx_mulc(Cpl<T>{x[u][0], -x[u][1]}, w);
          b2 = cx_mulc(Cpl<T>{x[u][2], -x[u][3]}, v);
          if (k == 0) b1.im = b2.im = 0;
        }
        const Cpl<T> e = {b1.re + b2.re, b1.im - b2.im};
        const Cpl<T> d = cx_mulc(Cpl<T>{b1.re - b2.re, b1.im + b2.im}, A.twn[k]);
        buf[(A.perm[k] << lc) + c] = Cpl<T>{e.re - d.im, e.im + d.re};  // e + i d
        if (k > 0 && m - k != k) buf[(A.perm[m - k] << lc) + c] = Cpl<T>{e.re + d.im, d.re - e.im};  // conj(e - i d)
      }
    }
  }
  __syncthreads();
  const ColsShift cm{lc};
  fft_all<true>(buf, A.F, A.F.l1 << lc, cm, A.fft, nt);
  const T* bt = reinterpret_cast<const T*>(smem);
  auto y_of = [&](int j, int cc) -> T {
    T y;
    if (four) {
      const int k = (j & 1) ? (n - 1 - j) >> 1 : j >> 1;
      const Cpl<T> z = buf[(k << lc) + cc], w = A.tw4b[k];
      y = (j & 1) ? (T)2 * (z.im * w.re - z.re * w.im) : (T)2 * (z.re * w.re + z.im * w.im);
    } else {
      const int t = kind == KIND_PP ? j : ((j & 1) ? n - 1 - (j >> 1) : (j >> 1));
      y = bt[(((t >> 1) << lc) + cc) * 2 + (t & 1)];
    }
    return neg_if(flip && (j & 1), y);
  };
  if (sk != 1) {
    double* dst = p3 + (live ? coff[c] : 0);
    for (int j0 = r0; j0 < n; j0 += ZLB * rs) {
      double old[ZLB];
#pragma unroll
      for (int u = 0; u < ZLB; ++u) {
        const int j = j0 + u * rs;
        old[u] = live && j < n ? dst[(long long)j * sk] : 0.0;
      }
#pragma unroll
      for (int u = 0; u < ZLB; ++u) {
        const int j = j0 + u * rs;
        if (j < n && live) dst[(long long)j * sk] = fma(to_double(y_of(j, c)), inv_theta, old[u]);
      }
    }
  } else {
    for (int i = threadIdx.x; i < n << lc; i += nt) {
      const int cc = i / n, j = i - cc * n;
      if (cc < ch.ncol) p3[coff[cc] + j] = fma(to_double(y_of(j, cc)), inv_theta, p3[coff[cc] + j]);
    }
  }
}

}  // namespace
}  // namespace snac
