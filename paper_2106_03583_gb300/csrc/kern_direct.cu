// Separable solve of the reduced equations (Eq. 9) for planes too large for one CTA's shared memory:
// three passes over the mode-space field, each reading and writing it once --
//   k_lines_fwd  transform along the uniform plane axis, planes -> spectral [q][n][kappa]
//   k_tri_*      one tridiagonal system per (q, kappa) along the other axis, in place
//   k_lines_bwd  inverse transform, spectral -> planes
// and the plan-side tables of the method (see direct_dev.cuh for the transforms and the systems).
#include <algorithm>
#include <cmath>
#include <vector>

#include "direct_dev.cuh"

namespace snac {
namespace {

constexpr int LNT = 256;  // threads of a line-transform CTA

// Shared memory of a line-transform CTA: C = 2^lc complex columns of F.n rows.
__host__ __device__ inline int line_s1(const FftTab& F, int lc) { return (F.l1 << lc) + 4; }
__host__ __device__ inline size_t line_smem(const FftTab& F, int lc, size_t w) {
  return 2 * w * (size_t)(F.n / F.l1) * line_s1(F, lc);
}

// Columns of a line CTA: besides the split of fft_dev.cuh, one in which a warp covers 4 columns x 8
// indices (32-byte segments of 8 lines' contiguous data).
struct ColsLine : ColsShift {
  __device__ __forceinline__ void split8(int t, int& idx, int& c) const {
    const int cl = lc < 2 ? lc : 2;
    const int lo = t & ((1 << cl) - 1), kk = (t >> cl) & 7, hi = t >> (cl + 3);
    const int ch = lc - cl;
    c = ((hi & ((1 << ch) - 1)) << cl) | lo;
    idx = ((hi >> ch) << 3) | kk;
  }
};

// Lines of one CTA: global line number g = q N + n; per line the plane base of q, its spectrum and n.
struct LineSet {
  long long* plane;  // q ncell, or -1 past the last line
  long long* spec;   // first element of the line's spectrum
  int* n;
};

template <typename T>
__device__ __forceinline__ long long line_off(const DirectArgs<T>& A, const LineSet& S, int l, int m) {
  const int n = S.n[l];
  const int b = A.nbm == 1 ? 0 : A.mblk[m];
  return S.plane[l] + A.base[n * A.nbm + b] + (long long)m * A.mstr[n];
}

// A line's place in the plane, kept by the thread that walks it: at(m) is the offset of cell m. Up to two
// blocks along m cost a selection; more take line_off.
template <typename T>
struct LineAt {
  long long o0, o1;
  int l;
  bool live;
  __device__ __forceinline__ LineAt(const DirectArgs<T>& A, const LineSet& S, int l_, int nlive) : l(l_), live(l_ < nlive) {
    const int n = live ? S.n[l] : 0;
    o0 = live ? S.plane[l] + A.base[n * A.nbm] : 0;
    o1 = live && A.nbm == 2 ? S.plane[l] + A.base[n * 2 + 1] : o0;
  }
  __device__ __forceinline__ long long at(const DirectArgs<T>& A, const LineSet& S, int str, int m) const {
    return A.nbm > 2 ? line_off(A, S, l, m) : (m < A.m1 ? o0 : o1) + (long long)m * str;
  }
};

template <typename T>
__device__ __forceinline__ int line_setup(const DirectArgs<T>& A, int lines, long long* plane, long long* spec, int* ln) {
  const int g0 = blockIdx.x * lines;
  const int total = A.nq * A.N;
  for (int l = threadIdx.x; l < lines; l += LNT) {
    const int g = g0 + l;
    const int q = g / A.N;
    plane[l] = g < total ? (long long)q * A.ncell : -1;
    ln[l] = g < total ? g - q * A.N : 0;
    spec[l] = (long long)q * A.ncell + A.soff + (long long)(g - q * A.N) * A.M;
  }
  __syncthreads();
  return g0;
}

constexpr int MAX_LINES = 64;
constexpr int LB = 4;  // loads of a batch in flight per thread

// Every thread keeps its column through all loops (LNT is a multiple of the threads of one index), so the line
// pointers are made once and an item costs no division. Bound by: FP64, its pipe (85 %, 512 x 512 x 256 cells 2.05 ms
// a launch); FP32, instruction issue and the latency of the passes (81 instructions per cell, down from 104: 0.25
// -> 0.21 ms, 2.6 TB/s).
template <typename T>
__global__ void __launch_bounds__(LNT, sizeof(T) == 4 ? 4 : 3) k_lines_fwd(const DirectArgs<T> A, int lc, const T* __restrict__ in,
                                                                         T* __restrict__ out) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ long long plane[MAX_LINES];
  __shared__ long long spec[MAX_LINES];
  __shared__ int ln[MAX_LINES];
  Cpl<T>* buf = reinterpret_cast<Cpl<T>*>(smem);
  T* bt = reinterpret_cast<T*>(smem);
  const ColsLine cm{{lc}};
  const int C = 1 << lc, M = A.M, kind = A.kind, s1 = line_s1(A.F, lc);
  const bool flip = flip_kind(kind), pair = A.cls == LINES_PAIR;
  const int lines = pair ? 2 * C : C;
  const int g0 = line_setup(A, lines, plane, spec, ln);
  const LineSet S{plane, spec, ln};
  const int nlive = min(lines, A.nq * A.N - g0);
  // LNT is a multiple of a column group's threads: a thread keeps its column(s) and walks the indices
  const int is = LNT >> lc;
  if (pair) {
    int i0, c;
    if (A.xl) cm.split8(threadIdx.x, i0, c);
    else cm.split(threadIdx.x, i0, c);
    const LineAt<T> pa(A, S, 2 * c, nlive), pb(A, S, 2 * c + 1, nlive);
    if (A.xl) {  // items: two consecutive cells of both lines of a column
      for (int h0 = i0; 2 * h0 < M; h0 += LB * is) {
        Cpl<T> a[LB], b[LB];
#pragma unroll
        for (int u = 0; u < LB; ++u) {
          const int m = 2 * (h0 + u * is);
          a[u] = b[u] = Cpl<T>{0, 0};
          if (m < M) {
            if (A.vec) {
              if (pa.live) a[u] = *reinterpret_cast<const Cpl<T>*>(in + pa.at(A, S, 1, m));
              if (pb.live) b[u] = *reinterpret_cast<const Cpl<T>*>(in + pb.at(A, S, 1, m));
            } else {
              if (pa.live) a[u] = Cpl<T>{in[pa.at(A, S, 1, m)], in[pa.at(A, S, 1, m + 1)]};
              if (pb.live) b[u] = Cpl<T>{in[pb.at(A, S, 1, m)], in[pb.at(A, S, 1, m + 1)]};
            }
          }
        }
#pragma unroll
        for (int u = 0; u < LB; ++u) {
          const int m = 2 * (h0 + u * is);
          if (m >= M) continue;
          a[u].im = neg_if(flip, a[u].im), b[u].im = neg_if(flip, b[u].im);
          buf[fft_row(pair_pos(kind, m, M), A.F, s1, C) + c] = Cpl<T>{a[u].re, b[u].re};
          buf[fft_row(pair_pos(kind, m + 1, M), A.F, s1, C) + c] = Cpl<T>{a[u].im, b[u].im};
        }
      }
    } else {  // the lines are adjacent in memory: one element of both lines of a column
      const int str = A.mstr[S.n[2 * c]], strb = A.mstr[S.n[2 * c + 1]];
      for (int m0 = i0; m0 < M; m0 += 2 * LB * is) {
        Cpl<T> v[2 * LB];
#pragma unroll
        for (int u = 0; u < 2 * LB; ++u) {
          const int m = m0 + u * is;
          v[u] = Cpl<T>{0, 0};
          if (m < M) {
            if (A.vec) {
              if (pa.live) v[u] = *reinterpret_cast<const Cpl<T>*>(in + pa.at(A, S, str, m));
            } else {
              if (pa.live) v[u].re = in[pa.at(A, S, str, m)];
              if (pb.live) v[u].im = in[pb.at(A, S, strb, m)];
            }
          }
        }
#pragma unroll
        for (int u = 0; u < 2 * LB; ++u) {
          const int m = m0 + u * is;
          if (m >= M) continue;
          v[u] = Cpl<T>{neg_if(flip && (m & 1), v[u].re), neg_if(flip && (m & 1), v[u].im)};
          buf[fft_row(pair_pos(kind, m, M), A.F, s1, C) + c] = v[u];
        }
      }
    }
  } else {
    // t_j and t_j' (j' = M/2 - 1 - j) from cells 2j, 2j+1, 2j', 2j'+1 of the column's line
    const int h = M / 2, items = (h + 1) / 2;
    int j0, c;
    if (A.xl) cm.split8(threadIdx.x, j0, c);
    else cm.split(threadIdx.x, j0, c);
    const LineAt<T> pa(A, S, c, nlive);
    const int str = A.mstr[S.n[c]];
    for (int j = j0; j < items; j += is) {
      const int jj = h - 1 - j;
      Cpl<T> p{0, 0}, r{0, 0};
      if (c < nlive) {
        p = Cpl<T>{in[pa.at(A, S, str, 2 * j)], in[pa.at(A, S, str, 2 * j + 1)]};
        r = Cpl<T>{in[pa.at(A, S, str, 2 * jj)], in[pa.at(A, S, str, 2 * jj + 1)]};
      }
      p.im = neg_if(flip, p.im), r.im = neg_if(flip, r.im);
      buf[fft_row(j, A.F, s1, C) + c] = cx_mul(Cpl<T>{p.re, r.im}, A.t4a[j]);
      buf[fft_row(jj, A.F, s1, C) + c] = cx_mul(Cpl<T>{r.re, p.im}, A.t4a[jj]);
    }
  }
  __syncthreads();
  fft_all<false>(buf, A.F, s1, cm, A.tw, LNT);
  if (pair) {
    int k0, c;
    cm.split8(threadIdx.x, k0, c);
    const bool la = 2 * c < nlive, lb = 2 * c + 1 < nlive;
    T* oa = out + (la ? spec[2 * c] : 0);
    T* ob = out + (lb ? spec[2 * c + 1] : 0);
    for (int k = k0; 2 * k <= M; k += is) {
      const Cpl<T> z1 = buf[fft_row(A.perm[k], A.F, s1, C) + c];
      const Cpl<T> z2 = k == 0 ? z1 : buf[fft_row(A.perm[M - k], A.F, s1, C) + c];
      Cpl<T> y1, y2;
      pair_post(kind, kind == KIND_PP ? Cpl<T>{1, 0} : A.w2n[k], z1, z2, y1, y2);
      const bool mirror = k > 0 && 2 * k < M;
      if (la) {
        oa[k] = y1.re;
        if (mirror) oa[M - k] = y2.re;
      }
      if (lb) {
        ob[k] = y1.im;
        if (mirror) ob[M - k] = y2.im;
      }
    }
  } else {
    const int h = M / 2, items = (h + 1) / 2;
    int k0, c;
    cm.split8(threadIdx.x, k0, c);
    T* o = out + (c < nlive ? spec[c] : 0);
    for (int k = c < nlive ? k0 : items; k < items; k += is) {
      const int kk = h - 1 - k;
      const Cpl<T> v = cx_mul(buf[fft_row(A.perm[k], A.F, s1, C) + c], A.t4b[k]);
      const Cpl<T> w = cx_mul(buf[fft_row(A.perm[kk], A.F, s1, C) + c], A.t4b[kk]);
      o[2 * k] = (T)2 * v.re;
      o[2 * k + 1] = (T)-2 * w.im;
      o[2 * kk] = (T)2 * w.re;
      o[2 * kk + 1] = (T)-2 * v.im;
    }
  }
}

template <typename T>
__global__ void __launch_bounds__(LNT, sizeof(T) == 4 ? 4 : 3) k_lines_bwd(const DirectArgs<T> A, int lc, const T* __restrict__ in,
                                                                         T* __restrict__ out) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ long long plane[MAX_LINES];
  __shared__ long long spec[MAX_LINES];
  __shared__ int ln[MAX_LINES];
  Cpl<T>* buf = reinterpret_cast<Cpl<T>*>(smem);
  const ColsLine cm{{lc}};
  const int C = 1 << lc, M = A.M, kind = A.kind, s1 = line_s1(A.F, lc);
  const bool flip = flip_kind(kind), pair = A.cls == LINES_PAIR;
  const int lines = pair ? 2 * C : C;
  const int g0 = line_setup(A, lines, plane, spec, ln);
  const LineSet S{plane, spec, ln};
  const int nlive = min(lines, A.nq * A.N - g0);
  const int is = LNT >> lc;
  if (pair) {
    int k0, c;
    cm.split8(threadIdx.x, k0, c);
    const bool la = 2 * c < nlive, lb = 2 * c + 1 < nlive;
    const T* ia = in + (la ? spec[2 * c] : 0);
    const T* ib = in + (lb ? spec[2 * c + 1] : 0);
    for (; 2 * k0 <= M; k0 += LB * is) {
      Cpl<T> x1[LB], x2[LB];
#pragma unroll
      for (int u = 0; u < LB; ++u) {
        const int k = k0 + u * is;
        x1[u] = x2[u] = Cpl<T>{0, 0};
        if (2 * k <= M) {
          const bool two = k > 0 && !(kind == KIND_PP && 2 * k == M);
          if (la) {
            x1[u].re = ia[k];
            if (two) x2[u].re = ia[M - k];
          }
          if (lb) {
            x1[u].im = ib[k];
            if (two) x2[u].im = ib[M - k];
          }
        }
      }
#pragma unroll
      for (int u = 0; u < LB; ++u) {
        const int k = k0 + u * is;
        if (2 * k > M) continue;
        Cpl<T> z1, z2;
        pair_pre(kind, kind == KIND_PP ? Cpl<T>{1, 0} : A.w2n[k], x1[u], x2[u], z1, z2);
        buf[fft_row(A.perm[k], A.F, s1, C) + c] = z1;
        if (k > 0 && 2 * k < M) buf[fft_row(A.perm[M - k], A.F, s1, C) + c] = z2;
      }
    }
  } else {
    const int h = M / 2, items = (h + 1) / 2;
    int j0, c;
    cm.split8(threadIdx.x, j0, c);
    for (int j = j0; j < items; j += is) {
      const int jj = h - 1 - j;
      Cpl<T> p{0, 0}, r{0, 0};
      if (c < nlive) {
        const T* i = in + spec[c];
        p = Cpl<T>{i[2 * j], i[2 * j + 1]};
        r = Cpl<T>{i[2 * jj], i[2 * jj + 1]};
      }
      const Cpl<T> v = cx_mul(Cpl<T>{p.re, r.im}, A.t4a[j]), w = cx_mul(Cpl<T>{r.re, p.im}, A.t4a[jj]);
      buf[fft_row(A.perm[j], A.F, s1, C) + c] = Cpl<T>{v.re, -v.im};  // forward = conj(inverse(conj))
      buf[fft_row(A.perm[jj], A.F, s1, C) + c] = Cpl<T>{w.re, -w.im};
    }
  }
  __syncthreads();
  fft_all<true>(buf, A.F, s1, cm, A.tw, LNT);
  if (pair) {
    int i0, c;
    if (A.xl) cm.split8(threadIdx.x, i0, c);
    else cm.split(threadIdx.x, i0, c);
    const LineAt<T> pa(A, S, 2 * c, nlive), pb(A, S, 2 * c + 1, nlive);
    if (A.xl) {
      for (int m = 2 * i0; m < M; m += 2 * is) {
        const Cpl<T> e = buf[fft_row(pair_pos(kind, m, M), A.F, s1, C) + c];
        Cpl<T> o = buf[fft_row(pair_pos(kind, m + 1, M), A.F, s1, C) + c];
        o = Cpl<T>{neg_if(flip, o.re), neg_if(flip, o.im)};
        if (A.vec) {
          if (pa.live) *reinterpret_cast<Cpl<T>*>(out + pa.at(A, S, 1, m)) = Cpl<T>{e.re, o.re};
          if (pb.live) *reinterpret_cast<Cpl<T>*>(out + pb.at(A, S, 1, m)) = Cpl<T>{e.im, o.im};
        } else {
          if (pa.live) {
            out[pa.at(A, S, 1, m)] = e.re;
            out[pa.at(A, S, 1, m + 1)] = o.re;
          }
          if (pb.live) {
            out[pb.at(A, S, 1, m)] = e.im;
            out[pb.at(A, S, 1, m + 1)] = o.im;
          }
        }
      }
    } else {
      const int str = A.mstr[S.n[2 * c]], strb = A.mstr[S.n[2 * c + 1]];
      for (int m = i0; m < M; m += is) {
        Cpl<T> v = buf[fft_row(pair_pos(kind, m, M), A.F, s1, C) + c];
        v = Cpl<T>{neg_if(flip && (m & 1), v.re), neg_if(flip && (m & 1), v.im)};
        if (A.vec) {
          if (pa.live) *reinterpret_cast<Cpl<T>*>(out + pa.at(A, S, str, m)) = v;
        } else {
          if (pa.live) out[pa.at(A, S, str, m)] = v.re;
          if (pb.live) out[pb.at(A, S, strb, m)] = v.im;
        }
      }
    }
  } else {
    const int h = M / 2, items = (h + 1) / 2;
    int k0, c;
    if (A.xl) cm.split8(threadIdx.x, k0, c);
    else cm.split(threadIdx.x, k0, c);
    const LineAt<T> pa(A, S, c, nlive);
    const int str = A.mstr[S.n[c]];
    for (int k = pa.live ? k0 : items; k < items; k += is) {
      const int kk = h - 1 - k;
      const Cpl<T> z = buf[fft_row(k, A.F, s1, C) + c], y = buf[fft_row(kk, A.F, s1, C) + c];
      const Cpl<T> v = cx_mul(Cpl<T>{z.re, -z.im}, A.t4b[k]), w = cx_mul(Cpl<T>{y.re, -y.im}, A.t4b[kk]);
      const T sg = flip ? (T)2 : (T)-2;  // cells 2k + 1 carry -2 Im, sign-flipped for DN
      out[pa.at(A, S, str, 2 * k)] = (T)2 * v.re;
      out[pa.at(A, S, str, 2 * k + 1)] = sg * w.im;
      out[pa.at(A, S, str, 2 * kk)] = (T)2 * w.re;
      out[pa.at(A, S, str, 2 * kk + 1)] = sg * v.im;
    }
  }
}

// Dense transform of DL lines x DK outputs per CTA of 256 threads: out[line][o] = sum_i in[line][i] mat[i][o].
// FWD: planes -> spectra; else spectra -> planes. 2 M FMA per cell and way. A warp covers 8 line groups x 4
// output groups, so that an input is one 128-byte shared read for 8 lanes of 16 bytes and the matrix entries
// are broadcasts; FP32 multiplies two lines per packed FMA. Two stages of DM terms, the next one's loads in
// flight. FP64 is bound by its pipe (92 % of it; 320 x 160 x 96 cells in three rectangles: both ways 1.28 ->
// 1.18 ms against 16 x 2 lanes per warp and one stage), FP32 by the latency of shared reads at 16 warps per SM
// (42 % of the FP32 rate; 336 x 192 x 150: both ways 0.33 -> 0.23 ms). Matrix entries stored as pairs: slower.
template <typename T>
struct DenseTile {
  // FP64: 16 outputs wide, so that no FP64 operation is spent on padding of common lengths
  static constexpr int V = 16 / sizeof(T), RL = 8, RO = sizeof(T) == 4 ? 4 : 1, DL = 16 * RL, DK = 16 * RO, DM = 16;
};

__device__ __forceinline__ void dense_fma(float (&acc)[8][4], const float (&a)[8], const float (&b)[4]) {
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const float2 bb = make_float2(b[j], b[j]);
#pragma unroll
    for (int i = 0; i < 8; i += 2) {
      const float2 r = __ffma2_rn(make_float2(a[i], a[i + 1]), bb, make_float2(acc[i][j], acc[i + 1][j]));
      acc[i][j] = r.x;
      acc[i + 1][j] = r.y;
    }
  }
}
__device__ __forceinline__ void dense_fma(double (&acc)[8][1], const double (&a)[8], const double (&b)[1]) {
#pragma unroll
  for (int i = 0; i < 8; ++i) acc[i][0] = fma(a[i], b[0], acc[i][0]);
}

template <typename T, bool FWD>
__global__ void __launch_bounds__(256, 2) k_dense(const DirectArgs<T> A, const T* __restrict__ in, T* __restrict__ out) {
  using D = DenseTile<T>;
  constexpr int V = D::V, RL = D::RL, RO = D::RO, DL = D::DL, DK = D::DK, DM = D::DM;
  struct alignas(16) Vec {
    T v[V];
  };
  __shared__ long long plane[DL];
  __shared__ long long spec[DL];
  __shared__ int ln[DL];
  __shared__ long long org[DL];  // a line's first input and its stride (one block along m)
  __shared__ int str[DL];
  __shared__ __align__(16) T as[2][DM][DL + V];
  __shared__ __align__(16) T bs[2][DM][DK];
  const int M = A.M;
  const long long total = (long long)A.nq * A.N, g0 = (long long)blockIdx.x * DL;
  for (int l = threadIdx.x; l < DL; l += 256) {
    const long long g = g0 + l;
    const int q = g < total ? (int)(g / A.N) : 0, n = g < total ? (int)(g - (long long)q * A.N) : 0;
    plane[l] = (long long)q * A.ncell;
    spec[l] = (long long)q * A.ncell + A.soff + (long long)n * M;
    ln[l] = n;
    org[l] = FWD ? plane[l] + A.base[n * A.nbm] : spec[l];
    str[l] = FWD ? A.mstr[n] : 1;
  }
  __syncthreads();
  const LineSet S{plane, spec, ln};
  const int nlive = (int)min((long long)DL, total - g0);
  const T* __restrict__ mat = FWD ? A.F1 : A.B1;
  const int o0 = blockIdx.y * DK;
  const int lane = threadIdx.x % 32, warp = threadIdx.x / 32;
  const int tx = (warp % 2) * 8 + lane % 8, ty = (warp / 2) * 4 + lane / 8;
  const bool along = !FWD || A.xl;  // the inputs of a line are contiguous
  const bool one = !FWD || A.nbm == 1;
  T acc[RL][RO];
#pragma unroll
  for (int i = 0; i < RL; ++i)
#pragma unroll
    for (int j = 0; j < RO; ++j) acc[i][j] = 0;
  constexpr int NA = DM * DL / 256, NB = DM * DK / 256;
  T ra[NA], rb[NB];
  auto fetch = [&](int m0) {
#pragma unroll
    for (int u = 0; u < NA; ++u) {
      const int t = threadIdx.x + u * 256;
      const int l = along ? t / DM : t % DL, m = m0 + (along ? t % DM : t / DL);
      ra[u] = (T)0;
      if (l < nlive && m < M) ra[u] = in[one ? org[l] + (long long)m * str[l] : line_off(A, S, l, m)];
    }
#pragma unroll
    for (int u = 0; u < NB; ++u) {
      const int t = threadIdx.x + u * 256, m = m0 + t / DK, o = o0 + t % DK;
      rb[u] = m < M && o < M ? mat[(long long)m * M + o] : (T)0;
    }
  };
  auto keep = [&](int st) {
#pragma unroll
    for (int u = 0; u < NA; ++u) {
      const int t = threadIdx.x + u * 256;
      if (along) as[st][t % DM][t / DM] = ra[u];
      else as[st][t / DL][t % DL] = ra[u];
    }
#pragma unroll
    for (int u = 0; u < NB; ++u) {
      const int t = threadIdx.x + u * 256;
      bs[st][t / DK][t % DK] = rb[u];
    }
  };
  fetch(0);
  int st = 0;
  for (int m0 = 0; m0 < M; m0 += DM, st ^= 1) {
    keep(st);  // (the other threads read this stage last before the previous barrier)
    __syncthreads();
    if (m0 + DM < M) fetch(m0 + DM);
#pragma unroll
    for (int k = 0; k < DM; ++k) {
      T a[RL], b[RO];
#pragma unroll
      for (int c = 0; c < RL / V; ++c) {
        const Vec v = *reinterpret_cast<const Vec*>(&as[st][k][V * tx + 16 * V * c]);
#pragma unroll
        for (int i = 0; i < V; ++i) a[V * c + i] = v.v[i];
      }
#pragma unroll
      for (int j = 0; j < RO; ++j) b[j] = bs[st][k][RO * ty + j];
      dense_fma(acc, a, b);
    }
  }
  const int o = o0 + RO * ty;
#pragma unroll
  for (int i = 0; i < RL; ++i) {
    const int l = V * tx + 16 * V * (i / V) + i % V;
    if (l >= nlive || o >= M) continue;
    const long long at = FWD ? spec[l] + o : line_off(A, S, l, o);
    if (RO == V && o + V <= M && (reinterpret_cast<size_t>(out + at) & 15) == 0 &&
        (FWD || line_off(A, S, l, o + V - 1) == at + V - 1)) {
      Vec v;
#pragma unroll
      for (int j = 0; j < V; ++j) v.v[j] = acc[i][j % RO];
      *reinterpret_cast<Vec*>(out + at) = v;
      continue;
    }
#pragma unroll
    for (int j = 0; j < RO; ++j)
      if (o + j < M) out[FWD ? at + j : line_off(A, S, l, o + j)] = acc[i][j];
  }
}

// The smoothest systems of an FP32 plan in FP64 arithmetic (FP32 right-hand side and solution). A
// rounded elimination leaves errors that differ from row to row, relative to the solution; the outer
// residual sees them times the row coupling (1e6 and more on a stretched axis), and the solution is
// largest where lambda + sigma is smallest. These few systems (list) therefore set the residual a
// correction step can reach: with all of them in FP32 the second step on the 1024 x 512 x 512 channel ends
// at 0.9-1.5e-10 relative residual, with the list in FP64 at 5e-11.
// ENDS: only the first and last unknowns, into the end vector of the interface systems, and num (tri_segment) of
// the pinned ones; pin, alpha, num: of the piece, IFACE_MAX_ENDS apart per wavenumber.
constexpr int LOW_KG = 8, LOW_R = 8;
template <bool ENDS>
__global__ void __launch_bounds__(512, 1) k_tri_low(const TriRow<double>* __restrict__ tri, const double* __restrict__ lam,
                                                  const double* __restrict__ sigma, double cscale, double scale,
                                                  const int* __restrict__ list, int nlist, int M, int N, int P,
                                                  long long ncell, int soff, int pin, const float* __restrict__ alpha,
                                                  float* __restrict__ num, float* __restrict__ x,
                                                  float* __restrict__ ends, int E, int e0, int e1) {
  extern __shared__ __align__(16) unsigned char smem[];
  const int kk = threadIdx.x % LOW_KG, seg = threadIdx.x / LOW_KG;
  const int k = blockIdx.x * LOW_KG + kk;
  const bool live = k < nlist;
  const int sys = live ? list[k] : 0;
  const int q = sys / M, kap = sys - q * M;
  float* col = x + (long long)q * ncell + soff + kap;
  const double tq = live ? -fma(sigma[q], cscale, lam[kap]) : 1.0;
  const bool pinned = pin && live && kap == 0;
  tri_segment<double, LOW_R>(tri, N, P, seg, kk, LOW_KG, true, live, tq, scale, pinned,
                             pinned && !ENDS ? (double)alpha[q * IFACE_MAX_ENDS] : 0.0, reinterpret_cast<double*>(smem),
                             [&](int n) { return (double)col[(long long)n * M]; },
                             [&](int n, double v) {
                               if (!ENDS) col[(long long)n * M] = (float)v;
                               else if (n == 0 && e0 >= 0) ends[(long long)q * E + e0 + kap] = (float)v;
                               else if (n == N - 1 && e1 >= 0) ends[(long long)q * E + e1 + kap] = (float)v;
                             },
                             [&](double v) {
                               if (ENDS) num[q * IFACE_MAX_ENDS] = (float)v;
                             });
}

// The elimination would be bound by arithmetic (14 operations per row, half of them for the pivot's reciprocal,
// which depends on the plan only), so the reciprocals are kept: [row of DirectTab::qrow][n][kappa], wavenumbers of
// equal sigma (q and n - q of the real DFT) sharing one set; that of a pinned unknown is kept as zero. The solve is
// then 5 operations per row. FP64 plans walk
// the rows twice (k_tri_pre, 48 bytes per cell; 512 x 512 x 256: 1.89 -> 0.69 ms, the FP64 pipe alone takes 0.53);
// FP32 plans take k_tri_scan, and k_tri_pre only for systems of more than 1024 rows.
template <typename T>
__global__ void __launch_bounds__(128) k_tri_factor(const TriRow<double>* __restrict__ tri, const double* __restrict__ lam,
                                                  const double* __restrict__ sigma, double cscale, int M, int N, int pin,
                                                  const int* __restrict__ qof, int rows, T* __restrict__ fac) {
  const long long sys = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (sys >= (long long)rows * M) return;
  const int r = (int)(sys / M), kap = (int)(sys - (long long)r * M);
  const double tq = -fma(sigma[qof[r]], cscale, lam[kap]);
  T* f = fac + (long long)r * N * M + kap;
  double g = 0;
  for (int n = 0; n < N; ++n) {
    const TriRow<double> w = tri[n];
    const double s = fma(w.lo, g, w.tau + tq);
    const double den = s + w.hi;
    const double inv = den > 0 ? 1.0 / den : 0.0;
    g = s * inv;
    f[(long long)n * M] = pin && kap == 0 && n == N - 1 ? (T)0 : (T)inv;
  }
}

constexpr int TRI_U = 8;  // rows whose loads are in flight per thread
template <typename T>
__global__ void __launch_bounds__(128, 8) k_tri_pre(const DirectArgs<T> A, const int* __restrict__ qrow,
                                                  const unsigned char* __restrict__ low, const T* __restrict__ fac,
                                                  const T* __restrict__ alpha, T* __restrict__ x) {
  const long long sys = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (sys >= (long long)A.nq * A.M || (sizeof(T) == 4 && low[sys])) return;
  const int q = (int)(sys / A.M), kap = (int)(sys - (long long)q * A.M);
  const int N = A.N, M = A.M;
  x += (long long)q * A.ncell + A.soff + kap;
  fac += (long long)qrow[q] * N * M + kap;
  const T sc = -A.scale;
  T d = 0;
  for (int n0 = 0; n0 < N; n0 += TRI_U) {
    T v[TRI_U], f[TRI_U];
#pragma unroll
    for (int u = 0; u < TRI_U; ++u) {
      const bool in = n0 + u < N;
      v[u] = in ? x[(long long)(n0 + u) * M] : (T)0;
      f[u] = in ? fac[(long long)(n0 + u) * M] : (T)0;
    }
#pragma unroll
    for (int u = 0; u < TRI_U; ++u) {
      if (n0 + u >= N) break;
      d = fma(A.tri[n0 + u].lo, d, sc * v[u]) * f[u];
      x[(long long)(n0 + u) * M] = d;
    }
  }
  if (A.pin && kap == 0) x[(long long)(N - 1) * M] = alpha[q * IFACE_MAX_ENDS];  // (zero so far: its f is zero)
  T y = 0;
  for (int n0 = (N - 1) / TRI_U * TRI_U; n0 >= 0; n0 -= TRI_U) {
    T v[TRI_U], f[TRI_U];
#pragma unroll
    for (int u = 0; u < TRI_U; ++u) {
      const bool in = n0 + u < N;
      v[u] = in ? x[(long long)(n0 + u) * M] : (T)0;
      f[u] = in ? fac[(long long)(n0 + u) * M] : (T)0;
    }
#pragma unroll
    for (int u = TRI_U - 1; u >= 0; --u) {
      if (n0 + u >= N) continue;
      y = fma(A.tri[n0 + u].hi * f[u], y, v[u]);
      x[(long long)(n0 + u) * M] = y;
    }
  }
}

// FP32 plans: the field is read and written once (12 bytes per cell instead of k_tri_pre's 24; FP64 would pay the
// 12 operations per row). Measured with the listed systems' k_tri_low: 512 x 512 x 256 cells 0.345 -> 0.262 ms,
// 1024 x 512 x 512 1.14 -> 0.81 ms (4.0 TB/s; stalls: barriers 3.1, memory 2.6 per issue, 58 % of the issue slots); 256 x 256 x 32 50 ->
// 47 us, 336 x 192 x 150 0.11 -> 0.085 ms against the segments eliminated without kept pivots. Two CTAs of 512
// threads per multiprocessor: four of 256 (shorter rows of systems) take 0.31 ms, one of 1024 0.29 ms.
// One thread per system and segment of TRI_R rows, which stay in its registers; with the pivots known, both
// sweeps are first-order recurrences, so a segment is an affine map of the value that enters it: the segments'
// maps are composed in order by the first segment's thread, then each thread runs its rows again from the right
// value, rounding as the sequential sweep does. All coefficients are >= 0. 2^lg systems per CTA.
// ENDS: only the first and last unknowns and num (see k_tri_ends), nothing is written to the field.
constexpr int SCAN_NT = 512, TRI_R = 16;
template <bool ENDS>
__global__ void __launch_bounds__(SCAN_NT, 2) k_tri_scan(const DirectArgs<float> A, int lg, int P, const int* __restrict__ qrow,
                                                        const unsigned char* __restrict__ low, const float* __restrict__ fac,
                                                        const float* __restrict__ alpha, float* __restrict__ x,
                                                        float* __restrict__ ends, int E, float* __restrict__ num) {
  constexpr int R = TRI_R;
  extern __shared__ __align__(16) unsigned char smem[];
  float2* lohi = reinterpret_cast<float2*>(smem);             // [P R] couplings
  float2* ex = lohi + P * R;                                  // [P][2^lg] segment maps, then entering values
  const int N = A.N, M = A.M, KG = 1 << lg;
  const int kk = threadIdx.x & (KG - 1), seg = threadIdx.x >> lg;
  const long long sys = ((long long)blockIdx.x << lg) + kk;
  const bool in = sys < (long long)A.nq * M;
  const bool live = in && !low[sys];  // (k_tri_low solves the others)
  const int q = in ? (int)(sys / M) : 0, kap = in ? (int)(sys - (long long)q * M) : 0;
  const bool pinned = live && A.pin && kap == 0;
  const int n0 = seg * R;
  float* col = x + (long long)q * A.ncell + A.soff + kap + (long long)n0 * M;
  const float* fc = fac + (long long)qrow[q] * N * M + kap + (long long)n0 * M;
  float v[R], f[R];
#pragma unroll
  for (int r = 0; r < R; ++r) {
    const bool ok = n0 + r < N;
    v[r] = ok && live ? col[(long long)r * M] : 0.0f;
    f[r] = ok && live ? fc[(long long)r * M] : 0.0f;
  }
  for (int n = threadIdx.x; n < P * R; n += blockDim.x) {
    const bool ok = n < N;
    lohi[n] = make_float2(ok ? A.tri[n].lo : 0.0f, ok ? A.tri[n].hi : 0.0f);
  }
  __syncthreads();
  float2* e = ex + threadIdx.x;
  float d = 0, a = 1;
#pragma unroll
  for (int r = 0; r < R; ++r) {
    const float lo = lohi[n0 + r].x;
    v[r] *= -A.scale;
    d = fma(lo, d, v[r]) * f[r];
    a *= lo * f[r];
  }
  *e = make_float2(d, a);
  __syncthreads();
  if (seg == 0) {
    float g = 0;
    for (int k = kk; k < P << lg; k += KG) {
      const float2 m = ex[k];
      ex[k].x = g;
      g = fma(m.y, g, m.x);
    }
  }
  __syncthreads();
  d = e->x;
#pragma unroll
  for (int r = 0; r < R; ++r) {
    d = fma(lohi[n0 + r].x, d, v[r]);
    if (n0 + r == N - 1 && pinned) {
      if (ENDS) num[q * IFACE_MAX_ENDS] = d;
      v[r] = ENDS ? 0.0f : alpha[q * IFACE_MAX_ENDS];
    } else {
      d *= f[r];
      v[r] = d;
    }
    if (ENDS && n0 + r == N - 1 && live && A.e1 >= 0) ends[(long long)q * E + A.e1 + kap] = v[r];
  }
  float y = 0, c = 1;
#pragma unroll
  for (int r = R - 1; r >= 0; --r) {
    const float h = lohi[n0 + r].y * f[r];
    y = fma(h, y, v[r]);
    c *= h;
  }
  *e = make_float2(y, c);
  __syncthreads();
  if (seg == 0) {
    float g = 0;
    for (int k = ((P - 1) << lg) + kk; k >= 0; k -= KG) {
      const float2 m = ex[k];
      ex[k].x = g;
      g = fma(m.y, g, m.x);
    }
    if (ENDS && live && A.e0 >= 0) ends[(long long)q * E + A.e0 + kap] = g;
  }
  if (ENDS) return;
  __syncthreads();
  y = e->x;
#pragma unroll
  for (int r = R - 1; r >= 0; --r) {
    y = fma(lohi[n0 + r].y * f[r], y, v[r]);
    if (live && n0 + r < N) col[(long long)r * M] = y;
  }
}

// Systems per CTA (log2) of k_tri_scan: 8 to 32, so that its rows are whole sectors; -1: too many segments.
inline int scan_lg(int P) {
  for (int lg = 5; lg >= 3; --lg)
    if (P << lg <= SCAN_NT) return lg;
  return -1;
}

template <bool ENDS>
void launch_scan(const DirectArgs<float>& A, int lg, const int* qrow, const unsigned char* low, const float* fac,
                 const float* alpha, float* x, float* ends, int E, float* num, cudaStream_t s) {
  const int P = (A.N + TRI_R - 1) / TRI_R;
  const long long sys = (long long)A.nq * A.M;
  const size_t smem = sizeof(float2) * ((size_t)P * TRI_R + ((size_t)P << lg));
  k_tri_scan<ENDS><<<(unsigned)((sys + (1 << lg) - 1) >> lg), P << lg, smem, s>>>(A, lg, P, qrow, low, fac, alpha, x, ends, E,
                                                                                  num);
}

// First and last unknowns of every system of a piece (the end values of the interface systems), from the
// kept pivots (the listed systems of an FP32 plan: k_tri_low). num: what the elimination leaves in the last row
// of the pinned systems (their last unknown is taken as zero).
template <typename T>
__global__ void __launch_bounds__(128, 8) k_tri_ends(const DirectArgs<T> A, const int* __restrict__ qrow,
                                                   const unsigned char* __restrict__ low, const T* __restrict__ fac,
                                                   const T* __restrict__ x, T* __restrict__ ends, int E,
                                                   T* __restrict__ num) {
  const long long sys = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (sys >= (long long)A.nq * A.M) return;
  const int q = (int)(sys / A.M), kap = (int)(sys - (long long)q * A.M);
  const int N = A.N, M = A.M;
  x += (long long)q * A.ncell + A.soff + kap;
  if (sizeof(T) == 4 && low[sys]) return;
  fac += (long long)qrow[q] * N * M + kap;
  const T sc = -A.scale;
  T d = 0, pi = 1, F = 0;
  for (int n0 = 0; n0 < N; n0 += TRI_U) {
    T v[TRI_U], f[TRI_U];
#pragma unroll
    for (int u = 0; u < TRI_U; ++u) {
      const bool in = n0 + u < N;
      v[u] = in ? x[(long long)(n0 + u) * M] : (T)0;
      f[u] = in ? fac[(long long)(n0 + u) * M] : (T)0;
    }
#pragma unroll
    for (int u = 0; u < TRI_U; ++u) {
      if (n0 + u >= N) break;
      const TriRow<T> w = A.tri[n0 + u];
      d = fma(w.lo, d, sc * v[u]);
      if (n0 + u == N - 1 && A.pin && kap == 0) num[q * IFACE_MAX_ENDS] = d;
      d *= f[u];
      F = fma(pi, d, F);
      pi *= w.hi * f[u];
    }
  }
  if (A.e0 >= 0) ends[(long long)q * E + A.e0 + kap] = F;
  if (A.e1 >= 0) ends[(long long)q * E + A.e1 + kap] = d;
}

template <typename T>
__global__ void __launch_bounds__(256) k_nonfinite(const T* __restrict__ v, long long n, int* __restrict__ flag) {
  bool bad = false;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
    bad = bad || !isfinite(v[i]);
  if (__syncthreads_or(bad) && threadIdx.x == 0) atomicOr(flag, 1);
}

// Complex columns per line CTA: about 32 KB of shared memory, 2 to 16 columns.
template <typename T>
int line_columns(const DirectArgs<T>& A) {
  int lc = 1;
  while (lc < 4 && ((size_t)A.F.n << (lc + 1)) * 2 * sizeof(T) <= 36 * 1024) ++lc;
  return lc;
}

template <typename T>
cudaError_t lines_t(snac_plan* P, const DirectArgs<T>& A, bool fwd, const T* in, T* out, cudaStream_t s) {
  if (A.cls == LINES_DENSE) {
    const double cells = (double)A.nq * A.M * A.N;
    LaunchScope ls(P, fwd ? K_LINES_FWD : K_LINES_BWD, 2.0 * sizeof(T) * cells, 2.0 * A.M * cells, s);
    const dim3 g((unsigned)(((long long)A.nq * A.N + DenseTile<T>::DL - 1) / DenseTile<T>::DL),
                 (unsigned)((A.M + DenseTile<T>::DK - 1) / DenseTile<T>::DK));
    if (fwd) k_dense<T, true><<<g, 256, 0, s>>>(A, in, out);
    else k_dense<T, false><<<g, 256, 0, s>>>(A, in, out);
    return cudaGetLastError();
  }
  const int lc = line_columns(A), lines = A.cls == LINES_PAIR ? 2 << lc : 1 << lc;
  const unsigned grid = (unsigned)(((long long)A.nq * A.N + lines - 1) / lines);
  const size_t smem = line_smem(A.F, lc, sizeof(T));
  const double cells = (double)A.nq * A.M * A.N;
  constexpr int kMax = 160 * 1024;  // the largest need (4096-point FP64 lines): function-wide, never lowered
  LaunchScope ls(P, fwd ? K_LINES_FWD : K_LINES_BWD, 2.0 * sizeof(T) * cells, (2.5 * std::log2((double)A.M) + 4.0) * cells, s);
  auto kern = fwd ? k_lines_fwd<T> : k_lines_bwd<T>;
  cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kMax);
  kern<<<grid, LNT, smem, s>>>(A, lc, in, out);
  return cudaGetLastError();
}

template <typename T>
cudaError_t tri_t(snac_plan* P, const DirectTab& D, const DirectArgs<T>& A, const T* alpha, T* u, cudaStream_t s) {
  const double cells = (double)A.nq * A.M * A.N;
  LaunchScope ls(P, K_TRI, 2.0 * sizeof(T) * cells, 20.0 * cells, s);
  const long long sys = (long long)A.nq * A.M;
  const unsigned g128 = (unsigned)((sys + 127) / 128);
  if constexpr (sizeof(T) == 4) {
    const int lsegs = (A.N + LOW_R - 1) / LOW_R;
    if (D.nlow)
      k_tri_low<false><<<(D.nlow + LOW_KG - 1) / LOW_KG, LOW_KG * lsegs, 7 * sizeof(double) * LOW_KG * lsegs, s>>>(
          (const TriRow<double>*)D.d_tri64, D.d_lam64, P->d_sigma64, D.cscale, D.cscale / D.theta, D.d_lowlist,
          D.nlow, A.M, A.N, lsegs, A.ncell, A.soff, A.pin, alpha, nullptr, u, nullptr, 0, -1, -1);
    const int lg = scan_lg((A.N + TRI_R - 1) / TRI_R);
    if (lg >= 0)
      launch_scan<false>(A, lg, P->direct.d_qrow, D.d_low, (const T*)D.d_fac, alpha, u, nullptr, 0, nullptr, s);
    else
      k_tri_pre<T><<<g128, 128, 0, s>>>(A, P->direct.d_qrow, D.d_low, (const T*)D.d_fac, alpha, u);
  } else {
    k_tri_pre<T><<<g128, 128, 0, s>>>(A, P->direct.d_qrow, nullptr, (const T*)D.d_fac, alpha, u);
  }
  return cudaGetLastError();
}

template <typename T>
cudaError_t direct_t(snac_plan* P, cudaStream_t s) {
  DirectPlan& D = P->direct;
  T* f = (T*)P->lev[0].d_f;
  T* u = (T*)P->lev[0].d_u;
  const int np = (int)D.pc.size();
  std::vector<DirectArgs<T>> A;
  for (const DirectTab& d : D.pc) A.push_back(direct_args<T>(P, d));
  cudaError_t e = cudaSuccess;
  for (int p = 0; p < np && e == cudaSuccess; ++p) e = lines_t(P, A[p], true, f, u, s);
  if (D.it.k) {
    for (int p = 0; p < np && e == cudaSuccess; ++p) {
      const DirectTab& d = D.pc[p];
      const double cells = (double)A[p].nq * d.M * d.N;
      LaunchScope ls(P, K_TRI, 2.0 * sizeof(T) * cells, 7.0 * cells, s);
      const long long sys = (long long)A[p].nq * d.M;
      if constexpr (sizeof(T) == 4) {
        const int lsegs = (d.N + LOW_R - 1) / LOW_R;
        if (d.nlow)
          k_tri_low<true><<<(d.nlow + LOW_KG - 1) / LOW_KG, LOW_KG * lsegs, 7 * sizeof(double) * LOW_KG * lsegs, s>>>(
              (const TriRow<double>*)d.d_tri64, d.d_lam64, P->d_sigma64, d.cscale, d.cscale / d.theta, d.d_lowlist,
              d.nlow, d.M, d.N, lsegs, A[p].ncell, A[p].soff, A[p].pin, nullptr, (T*)D.it.d_num + p, u, (T*)D.it.d_ends, D.it.E,
              A[p].e0, A[p].e1);
      }
      bool done = false;
      if constexpr (sizeof(T) == 4) {
        const int lg = scan_lg((d.N + TRI_R - 1) / TRI_R);
        done = lg >= 0;
        if (done)
          launch_scan<true>(A[p], lg, D.d_qrow, d.d_low, (const T*)d.d_fac, nullptr, u, (T*)D.it.d_ends, D.it.E,
                            (T*)D.it.d_num + p, s);
      }
      if (!done)
        k_tri_ends<T><<<(unsigned)((sys + 127) / 128), 128, 0, s>>>(A[p], D.d_qrow, d.d_low, (const T*)d.d_fac, u,
                                                                   (T*)D.it.d_ends, D.it.E, (T*)D.it.d_num + p);
      e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = launch_iface(P, s);
  }
  for (int p = 0; p < np && e == cudaSuccess; ++p)
    e = tri_t<T>(P, D.pc[p], A[p], D.it.ns ? (const T*)D.it.d_alpha + p : nullptr, u, s);
  for (int p = 0; p < np && e == cudaSuccess; ++p) e = lines_t(P, A[p], false, (const T*)u, f, s);
  return e;
}

}  // namespace

cudaError_t launch_nonfinite(snac_plan* P, const void* v, long long n, cudaStream_t s) {
  P->h_check[0] = 0;
  if (P->precision == SNAC_FP64) k_nonfinite<double><<<4 * P->sms, 256, 0, s>>>((const double*)v, n, P->dh_check);
  else k_nonfinite<float><<<4 * P->sms, 256, 0, s>>>((const float*)v, n, P->dh_check);
  return cudaGetLastError();
}

cudaError_t launch_tri_factor(snac_plan* P, const DirectTab& D, const int* d_qof, int rows, cudaStream_t s) {
  const bool f64 = P->precision == SNAC_FP64;
  const TriRow<double>* tri = (const TriRow<double>*)(f64 ? D.d_tri : (void*)D.d_tri64);
  const double* lam = f64 ? (const double*)D.d_lam : D.d_lam64;
  const unsigned grid = (unsigned)(((long long)rows * D.M + 127) / 128);
  if (f64) k_tri_factor<double><<<grid, 128, 0, s>>>(tri, lam, P->d_sigma64, D.cscale, D.M, D.N, D.pin, d_qof, rows, (double*)D.d_fac);
  else k_tri_factor<float><<<grid, 128, 0, s>>>(tri, lam, P->d_sigma64, D.cscale, D.M, D.N, D.pin, d_qof, rows, (float*)D.d_fac);
  return cudaGetLastError();
}

cudaError_t launch_direct(snac_plan* P, cudaStream_t s) {
  return P->precision == SNAC_FP64 ? direct_t<double>(P, s) : direct_t<float>(P, s);
}

}  // namespace snac
