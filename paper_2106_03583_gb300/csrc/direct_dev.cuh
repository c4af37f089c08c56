// Separable solve of the reduced equations (Eq. 9) on an assembled rectangle: device code.
//
// When the blocks of a plan assemble into a full rectangle, the reduced operator of every wavenumber
// is A_x + A_y + sigma_q with one-dimensional A_x, A_y. If one of the two plane axes is uniform, the
// real-to-real transform of its boundary pair diagonalises it (the same Table 1 kinds as along the
// homogeneous axis), and what is left is one tridiagonal system along the other axis per
// (wavenumber, transform slot): an exact solve of about 40 operations per cell in place of several
// V-cycles. "m" numbers cells along the transformed axis (M of them), "n" along the tridiagonal one
// (N); spectral slot kappa stands for one eigenvector of the transformed axis.
//
// Layouts of several such rectangles (pieces) that meet along parts of their first or last rows are solved
// piece by piece with Neumann faces there; the fluxes through the shared faces are the unknowns of a dense
// system per wavenumber, whose right-hand side needs only the first and last rows of the pieces' solutions.
// So a solve is: transforms, end values, interface systems (fluxes added to the end rows), tridiagonal
// solves, inverse transforms.
//
// Transforms work on complex columns of a shared-memory buffer (fft_dev.cuh):
//   pair kinds (PP, NN, DD): column c holds lines 2c and 2c+1 as real and imaginary part of one
//       length-M FFT; with Z_k = A_k + i B_k the two spectra separate by additions. PP is kept at twice
//       its usual scale; NN uses Makhoul's order v_t = x_2t | x_2(M-1-t)+1 and DD is NN of (-1)^m x_m
//       with its slots in the NN numbering (slot kappa = DST-II index M-1-kappa).
//   DCT-IV kinds (ND; DN = ND of (-1)^m x_m, slots reversed likewise): column c holds line c as a
//       half-length sequence t_j = (x_2j + i x_M-1-2j) e^{-i pi (4j+1)/4M}.
// Forward then inverse multiplies by 2 M for every kind; the tridiagonal solve divides by it.
//   dense (an axis that is not uniform, or a length with another prime factor; planes of several passes):
//       the eigenvectors of the one-dimensional operator, one M x M matrix product per line and way.
//
// Tridiagonal systems: (lo + hi + tau) u_n - lo u_{n-1} - hi u_{n+1} = -f_n / 2M with couplings lo, hi
// >= 0 and tau = -lambda_kappa - sigma_q + (Dirichlet face terms) >= 0. Elimination carries the row
// sums (tau) instead of the diagonal, so that every operation adds or multiplies non-negative numbers:
// no cancellation, the factors are accurate to a few units in the last place of the working type even
// where the system is nearly singular, and an exactly singular one (all tau = 0) ends in an exactly zero
// pivot, whose unknown is set to zero (the caller fixes the mean). A piece of several without a Dirichlet face, in
// a plan with small shifts, has the last unknown of its slot 0 given (pinned): its value alpha comes from the
// interface system.
#pragma once

#include <algorithm>

#include "fft_dev.cuh"

namespace snac {
namespace {

enum { LINES_PAIR = 0, LINES_DCT4 = 1, LINES_DENSE = 2 };

// One row of the tridiagonal axis: couplings, face term, and lo / hi (0 where hi = 0).
template <typename T>
struct alignas(4 * sizeof(T)) TriRow {
  T lo, hi, tau, ratio;
};

template <typename T>
struct DirectArgs {
  FftTab F;
  int M, N, cls, kind;
  int nq;                  // wavenumbers held
  const Cpl<T>* tw;        // e^{-2 pi i k / F.n}
  const Cpl<T>* w2n;       // e^{-i pi k / 2M}, k = 0..M (pair kinds)
  const Cpl<T>* t4a;       // e^{-i pi (4j+1) / 4M} (DCT-IV kinds)
  const Cpl<T>* t4b;       // e^{-i pi k / M}
  const int* perm;         // row of frequency k
  const T* lam;            // eigenvalue of slot kappa (<= 0), times cscale
  const TriRow<T>* tri;    // [N], times cscale
  const T* sigma;          // per wavenumber
  int pin;                 // slot 0 is pinned
  long long ncell;
  int soff;                // the piece's first spectral element within a plane
  int e0, e1;              // where its first / last row's values start in the end vector, -1: not needed
  T cscale;                // power of two that brings the couplings of tri (and lam) to about 1
  T scale;                 // cscale / theta (2M, dense: 1)
  const T* F1;             // LINES_DENSE: matrices [m][kappa], [kappa][m]
  const T* B1;
  // plane offset of (m, n): base[n nbm + mblk[m]] + m mstr[n]
  const int* base;
  const int* mblk;
  const int* mstr;
  int nbm, m1, xl, vec;    // m1: first m of the second block (M: one block); xl: the transformed axis is the
                           // contiguous one; vec: pairs may be loaded as vectors
};

template <typename T>
inline DirectArgs<T> direct_args(const snac_plan* P, const DirectTab& D) {
  DirectArgs<T> A{};
  const IfaceTab& I = P->direct.it;
  A.e0 = A.e1 = -1;
  for (int u = 0; u < I.nends; ++u)
    if (&P->direct.pc[I.ep[u]] == &D) (I.ee[u] == 0 ? A.e0 : A.e1) = I.eo[u];
  A.soff = D.soff;
  A.pin = D.pin;
  A.F = D.fft;
  A.M = D.M;
  A.N = D.N;
  A.cls = D.cls;
  A.kind = D.kind;
  A.nq = P->nz;
  A.tw = (const Cpl<T>*)D.d_tw;
  A.w2n = A.tw + D.w2n;
  A.t4a = A.tw + D.t4a;
  A.t4b = A.tw + D.t4b;
  A.perm = D.d_perm;
  A.lam = (const T*)D.d_lam;
  A.tri = (const TriRow<T>*)D.d_tri;
  if constexpr (sizeof(T) == 8) A.sigma = P->d_sigma64;
  else A.sigma = P->d_sigma32;
  A.ncell = P->lev[0].ncell;
  A.cscale = (T)D.cscale;
  A.scale = (T)(D.cscale / D.theta);
  A.F1 = (const T*)D.d_F;
  A.B1 = (const T*)D.d_B;
  A.base = D.d_base;
  A.mblk = D.d_mblk;
  A.mstr = D.d_mstr;
  A.nbm = D.nbm;
  A.m1 = D.m1;
  A.xl = D.xl;
  A.vec = D.vec;
  return A;
}

template <typename T>
struct IfaceArgs {
  int k, kk, E, ns, qs;             // qs: wavenumber whose whole system is singular (the last equation is implied)
  int sp[IFACE_MAX_ENDS];
  int nends, eo[IFACE_MAX_ENDS + 1];
  int row[IFACE_MAX_ENDS];          // first spectral element of every end row within a plane
  const double* Y;
  const T* Z;
  const double* KT;
  const int* qrow;
  T* ends;
  T* alpha;
  T* num;
};

template <typename T>
inline IfaceArgs<T> iface_args(const snac_plan* P) {
  const IfaceTab& I = P->direct.it;
  IfaceArgs<T> A{};
  A.k = I.k;
  A.kk = I.kk;
  A.E = I.E;
  A.ns = I.ns;
  A.qs = I.qs;
  A.nends = I.nends;
  for (int u = 0; u < I.nends; ++u) {
    const DirectTab& D = P->direct.pc[I.ep[u]];
    A.eo[u] = I.eo[u];
    A.row[u] = D.soff + (I.ee[u] ? (D.N - 1) * D.M : 0);
  }
  A.eo[I.nends] = I.E;
  for (int a = 0; a < I.ns; ++a) A.sp[a] = I.sp[a];
  A.Y = I.d_Y;
  A.Z = (const T*)I.d_Z;
  A.KT = I.d_KT;
  A.qrow = P->direct.d_qrow;
  A.ends = (T*)I.d_ends;
  A.alpha = (T*)I.d_alpha;
  A.num = (T*)I.d_num;
  return A;
}

// out[j] = sum_e A[e ld + j] x[e] for j < n by a CTA of nt threads (part: nt values); x in shared memory.
template <typename TA>
__device__ void gemv_cols(const TA* __restrict__ A, int ld, int n, int E, const TA* __restrict__ x, TA* __restrict__ out,
                          TA* __restrict__ part, int nt) {
  const int np = (n + 31) & ~31, tid = threadIdx.x;
  if (np <= nt) {  // the rows e split over nt / np groups of threads
    const int G = nt / np, g = tid / np, j = tid - g * np;
    TA acc = 0;
    if (g < G && j < n) {
#pragma unroll 16
      for (int e = g; e < E; e += G) acc = fma(A[(long long)e * ld + j], x[e], acc);
    }
    part[tid] = acc;
    __syncthreads();
    if (tid < n) {
      TA s = 0;
      for (int q = 0; q < G; ++q) s += part[q * np + tid];
      out[tid] = s;
    }
  } else {
    for (int j = tid; j < n; j += nt) {
      TA acc = 0;
#pragma unroll 16
      for (int e = 0; e < E; ++e) acc = fma(A[(long long)e * ld + j], x[e], acc);
      out[j] = acc;
    }
  }
  __syncthreads();
}

// The fluxes of wavenumber q from its end values: jumps of u across the interface cells, the dense system,
// and what the fluxes add to the end rows' right-hand sides (add(e, v)); num, alpha: the pinned pieces'
// eliminated last right-hand sides and unknowns (by piece). The jumps are differences of nearly equal end values and K^-1 damps their smooth
// part by the pieces' size in cells, so both products are formed in FP64 in every plan (in FP32 their
// rounding left a second correction step at 1e-9 .. 2e-8 of ||f|| on the L-shaped 512 x 512 x 128 duct).
// work (doubles, shared): ends (complete), y, phi, part: E + 2 kk + nt.
template <typename T, typename Add>
__device__ void iface_solve(const IfaceArgs<T>& I, int q, double* work, const T* num, T* alpha, int nt, Add&& add) {
  double* ends = work;
  double* y = ends + I.E;
  double* phi = y + I.kk;
  double* part = phi + I.kk;
  gemv_cols(I.Y, I.kk, I.k, I.E, ends, y, part, nt);
  if ((int)threadIdx.x < I.ns) {
    const int a = threadIdx.x;
    y[I.k + a] = q == I.qs && a == I.ns - 1 ? 0.0 : (double)num[I.sp[a]];
  }
  __syncthreads();
  gemv_cols(I.KT + (long long)I.qrow[q] * I.kk * I.kk, I.kk, I.kk, I.kk, y, phi, part, nt);
  if ((int)threadIdx.x < I.ns) alpha[I.sp[threadIdx.x]] = (T)phi[I.k + threadIdx.x];
  T* ph = reinterpret_cast<T*>(part);  // (kk <= 1040 values of T fit in nt doubles)
  for (int j = threadIdx.x; j < I.k; j += nt) ph[j] = (T)phi[j];
  __syncthreads();
  for (int e = threadIdx.x; e < I.E; e += nt) {
    T acc = 0;
#pragma unroll 16
    for (int j = 0; j < I.k; ++j) acc = fma(I.Z[(long long)j * I.E + e], ph[j], acc);
    add(e, acc);
  }
  __syncthreads();
}

// Two spectra from one pair column: z1 = Z_k, z2 = Z_{M-k}; slots k -> y1 (line a, line b), M-k -> y2.
template <typename T>
__device__ __forceinline__ void pair_post(int kind, Cpl<T> w, Cpl<T> z1, Cpl<T> z2, Cpl<T>& y1, Cpl<T>& y2) {
  const T ar = z1.re + z2.re, ai = z1.im - z2.im, br = z1.im + z2.im, bi = z2.re - z1.re;
  if (kind == KIND_PP) {
    y1 = {ar, br};
    y2 = {ai, bi};
  } else {
    y1 = {w.re * ar - w.im * ai, w.re * br - w.im * bi};
    y2 = {-w.im * ar - w.re * ai, -w.im * br - w.re * bi};
  }
}

// The inverse: slots k, M-k of both lines -> Z_k, Z_{M-k} (k = 0: x2 is taken as zero by the caller).
template <typename T>
__device__ __forceinline__ void pair_pre(int kind, Cpl<T> w, Cpl<T> x1, Cpl<T> x2, Cpl<T>& z1, Cpl<T>& z2) {
  T ar = x1.re, ai = x2.re, br = x1.im, bi = x2.im;
  if (kind != KIND_PP) {
    ar = w.re * x1.re - w.im * x2.re;
    ai = -w.re * x2.re - w.im * x1.re;
    br = w.re * x1.im - w.im * x2.im;
    bi = -w.re * x2.im - w.im * x1.im;
  }
  z1 = {ar - bi, ai + br};
  z2 = {ar + bi, br - ai};
}

// Natural row of cell m of a pair column.
__device__ __forceinline__ int pair_pos(int kind, int m, int M) {
  return kind == KIND_PP ? m : ((m & 1) ? M - 1 - (m >> 1) : m >> 1);
}
__device__ __forceinline__ bool flip_kind(int kind) { return kind == KIND_DD || kind == KIND_DN; }

__device__ __forceinline__ float tri_recip(float x) { return __fdividef(1.0f, x); }
__device__ __forceinline__ double tri_recip(double x) { return recip(x); }

// R consecutive rows of a tridiagonal system per thread, P threads per system (segments; the first
// segment is padded in front by identity rows, so the last one ends at row N - 1). Each thread
// eliminates its rows to u_r = D_r + c_r u_{r+1} + a_r u_{-1} (u_{-1}: the previous segment's last
// unknown), the segments' last unknowns form a tridiagonal system of P rows that the first segment's
// thread solves, and each thread substitutes back. load(n) gives the right-hand side, store(n, u)
// takes the solution; ex: 7 x P x kg values, this system's column kk. Every thread of the CTA calls it
// (three barriers). tq = -lambda - sigma >= 0; pin: the last unknown is alpha, and num takes what its row is
// left with by the elimination; an exactly singular system that is not pinned ends in zero.
// `act` is false for threads past the last segment, which only take part in the barriers; `live`
// for those with a system to solve.
template <typename T, int R, typename Load, typename Store, typename Num>
__device__ __forceinline__ void tri_segment(const TriRow<T>* __restrict__ tri, int N, int P, int seg, int kk, int kg,
                                            bool act, bool live, T tq, T scale, bool pin, T alpha, T* __restrict__ ex,
                                            Load&& load, Store&& store, Num&& num) {
  const int n0 = seg * R - (P * R - N);
  T D[R], c[R];
#pragma unroll
  for (int r = 0; r < R; ++r) D[r] = live && n0 + r >= 0 ? load(n0 + r) : (T)0;
  T a = 1, sl = 0, dp = 0, pi = 1, F = 0, H = 0;
#pragma unroll
  for (int r = 0; r < R; ++r) {
    TriRow<T> w{0, 0, 1, 0};
    if (n0 + r >= 0) {
      w = tri[n0 + r];
      w.tau += tq;
    }
    const T la = w.lo * a, ls = fma(w.lo, sl, w.tau);
    const T den = la + ls + w.hi;
    // (a pinned last row stays as it is: num and the segments' system need it unscaled)
    const T inv = pin && r == R - 1 && seg == P - 1 ? (T)1 : den > (T)0 ? tri_recip(den) : (T)0;
    c[r] = w.hi * inv;
    a = la * inv;
    sl = ls * inv;
    dp = fma(w.lo, dp, -scale * D[r]) * inv;
    D[r] = dp;
    if (r < R - 1) {
      F = fma(pi, dp, F);
      H = fma(pi, sl, H);
      pi *= c[r];
    }
  }
  const int st = P * kg;
  T* e = ex + seg * kg + kk;
  if (act) {
    e[0] = dp;
    e[st] = c[R - 1];
    e[2 * st] = a;
    e[3 * st] = sl;
    e[4 * st] = F;
    e[5 * st] = pi;
    e[6 * st] = H;
  }
  __syncthreads();
  if (act && seg == 0) {
    T* z = ex + kk;
    T g = 0, y = 0;
    for (int s = 0; s < P; ++s) {
      const int o = s * kg;
      const bool more = s + 1 < P;
      const T cs = z[o + st];
      const T lo = z[o + 2 * st];
      const T hi = more ? cs * z[o + kg + 5 * st] : (T)0;
      const T tau = more ? fma(cs, z[o + kg + 6 * st], z[o + 3 * st]) : z[o + 3 * st];
      const T d = more ? fma(cs, z[o + kg + 4 * st], z[o]) : z[o];
      const T sum = fma(lo, g, tau);
      const T den = sum + hi;
      const T inv = den > (T)0 ? tri_recip(den) : (T)0;
      g = sum * inv;
      y = fma(lo, y, d);
      if (pin && !more) {
        num(y);
        y = alpha;
      } else {
        y *= inv;
      }
      z[o] = y;
      z[o + st] = hi * inv;
    }
    for (int s = P - 2; s >= 0; --s) {
      const int o = s * kg;
      y = fma(z[o + st], y, z[o]);
      z[o] = y;
    }
  }
  __syncthreads();
  T x = act ? e[0] : (T)0;
  T aa = act && seg > 0 ? e[-kg] : (T)0;
  __syncthreads();  // ex is free for the next round
#pragma unroll
  for (int r = 0; r < R - 1; ++r) {
    const T ra = n0 + r >= 0 ? tri[n0 + r].ratio : (T)0;
    aa *= ra * c[r];
    D[r] += aa;
  }
  if (live && n0 + R - 1 >= 0) store(n0 + R - 1, x);
#pragma unroll
  for (int r = R - 2; r >= 0; --r) {
    x = fma(c[r], x, D[r]);
    if (live && n0 + r >= 0) store(n0 + r, x);
  }
}

// Shared memory of a whole-plane solve: the buffer, then the exchange of the tridiagonal segments.
constexpr int PLANE_R = 8;  // rows per thread of the tridiagonal phase

struct PlaneShape {
  int cols, rp, s1;
  size_t buf;  // elements of the buffer (real)
};
__host__ __device__ inline PlaneShape plane_shape(const FftTab& F, int M, int N, int cls) {
  PlaneShape s;
  s.cols = cls == LINES_PAIR ? (N + 1) / 2 : N;
  s.rp = s.cols | 1;
  s.s1 = F.l1 * s.rp;
  s.s1 += (1 - s.s1) & 15;  // consecutive slots of the first radix on different banks
  s.buf = 2 * (size_t)(F.n / F.l1) * s.s1;
  return s;
}
// Elements of shared memory of a whole-plane solve: the pieces' buffers, the exchange of the tridiagonal
// segments, the pinned pieces' unknowns and right-hand sides, and (doubles) the work space of an interface solve.
inline size_t onchip_elements(size_t buffers, int nt) {
  return ((buffers + 1) & ~(size_t)1) + 7 * (size_t)nt + 2 * IFACE_MAX_ENDS;
}
inline size_t iface_doubles(int E, int kk, int nt) {
  return E ? E + 2 * (size_t)kk + std::max((size_t)nt, (size_t)kk) : 0;
}

template <typename T>
struct PlaneArgs {
  int np;
  const DirectArgs<T>* pc;   // device table
  const unsigned* celloff;   // per plane cell: element of the shared buffers | sign flip << 31
  long long ncell;
  size_t buffers;            // elements of all pieces' buffers (even)
  IfaceArgs<T> I;
};

template <typename T>
inline PlaneArgs<T> plane_args(const snac_plan* P) {
  PlaneArgs<T> A{};
  A.np = (int)P->direct.pc.size();
  A.pc = (const DirectArgs<T>*)P->direct.d_args;
  A.celloff = P->direct.d_celloff;
  A.ncell = P->lev[0].ncell;
  for (const DirectTab& d : P->direct.pc) A.buffers += plane_shape(d.fft, d.M, d.N, d.cls).buf;
  A.buffers = (A.buffers + 1) & ~(size_t)1;
  A.I = iface_args<T>(P);
  return A;
}

// Planes to spectra of one piece in its buffer (complete on entry, behind a barrier on return).
template <typename T>
__device__ void piece_forward(const DirectArgs<T>& A, const PlaneShape& S, Cpl<T>* buf, int nt) {
  const ColsAny cm{S.cols, S.rp, recip16(S.cols)};
  const int M = A.M, kind = A.kind;
  const bool pair = A.cls == LINES_PAIR;
  if (!pair) {
    for (int t = threadIdx.x; t < A.F.n * S.cols; t += nt) {
      int j, c;
      cm.split(t, j, c);
      const int o = fft_row(j, A.F, S.s1, S.rp) + c;
      buf[o] = cx_mul(buf[o], A.t4a[j]);
    }
    __syncthreads();
  }
  fft_all<false>(buf, A.F, S.s1, cm, A.tw, nt);
  if (pair) {
    for (int t = threadIdx.x; t < (M / 2 + 1) * S.cols; t += nt) {
      int k, c;
      cm.split(t, k, c);
      const int o1 = fft_row(A.perm[k], A.F, S.s1, S.rp) + c;
      const int o2 = k == 0 ? o1 : fft_row(A.perm[M - k], A.F, S.s1, S.rp) + c;
      Cpl<T> y1, y2;
      pair_post(kind, kind == KIND_PP ? Cpl<T>{1, 0} : A.w2n[k], buf[o1], buf[o2], y1, y2);
      if (o2 != o1) buf[o2] = y2;
      buf[o1] = y1;
    }
  } else {
    for (int t = threadIdx.x; t < A.F.n * S.cols; t += nt) {
      int k, c;
      cm.split(t, k, c);
      const int o = fft_row(A.perm[k], A.F, S.s1, S.rp) + c;
      const Cpl<T> v = cx_mul(buf[o], A.t4b[k]);
      buf[o] = Cpl<T>{(T)2 * v.re, (T)-2 * v.im};
    }
  }
  __syncthreads();
}

// Where slot kappa of a piece stands in its buffer: element o + n ns for row n.
template <typename T>
__device__ __forceinline__ int slot_at(const DirectArgs<T>& A, const PlaneShape& S, int kap) {
  if (A.cls == LINES_PAIR) return 2 * fft_row(A.perm[kap], A.F, S.s1, S.rp);
  return 2 * fft_row(A.perm[(kap & 1) ? (A.M - 1 - kap) >> 1 : kap >> 1], A.F, S.s1, S.rp) + (kap & 1);
}

// The tridiagonal systems of one piece; ENDS: only the first and last rows' solutions, into the end vector, and
// the pinned system's eliminated last right-hand side (*num).
template <typename T, bool ENDS>
__device__ void piece_tri(const DirectArgs<T>& A, const PlaneShape& S, T* bt, T sg, T alpha, T* ex, double* ends, T* num, int nt) {
  const int N = A.N, M = A.M;
  const int P = (N + PLANE_R - 1) / PLANE_R, kg = nt / P;
  const int seg = (int)threadIdx.x / kg, kk = threadIdx.x - seg * kg;
  const bool mine = seg < P;
  const int ns = A.cls == LINES_PAIR ? 1 : 2;
  for (int k0 = 0; k0 < M; k0 += kg) {
    const int kap = k0 + kk;
    const bool live = mine && kap < M;
    int o = 0;
    T tq = 0;
    if (live) {
      tq = -fma(sg, A.cscale, A.lam[kap]);
      o = slot_at(A, S, kap);
    }
    tri_segment<T, PLANE_R>(A.tri, N, P, mine ? seg : 0, kk, kg, mine, live, tq, A.scale, A.pin && live && kap == 0, alpha, ex,
                            [&](int n) { return bt[o + n * ns]; },
                            [&](int n, T v) {
                              if (!ENDS) {
                                bt[o + n * ns] = v;
                              } else {
                                if (n == 0 && A.e0 >= 0) ends[A.e0 + kap] = v;
                                if (n == N - 1 && A.e1 >= 0) ends[A.e1 + kap] = v;
                              }
                            },
                            [&](T v) {
                              if (ENDS) *num = v;
                            });
  }
  __syncthreads();
}

// Spectra back to planes of one piece.
template <typename T>
__device__ void piece_backward(const DirectArgs<T>& A, const PlaneShape& S, Cpl<T>* buf, int nt) {
  const ColsAny cm{S.cols, S.rp, recip16(S.cols)};
  const int M = A.M, kind = A.kind;
  const bool pair = A.cls == LINES_PAIR;
  if (pair) {
    for (int t = threadIdx.x; t < (M / 2 + 1) * S.cols; t += nt) {
      int k, c;
      cm.split(t, k, c);
      const int o1 = fft_row(A.perm[k], A.F, S.s1, S.rp) + c;
      const int o2 = k == 0 ? o1 : fft_row(A.perm[M - k], A.F, S.s1, S.rp) + c;
      const Cpl<T> x1 = buf[o1];
      const Cpl<T> x2 = k == 0 || (kind == KIND_PP && 2 * k == M) ? Cpl<T>{0, 0} : buf[o2];
      Cpl<T> z1, z2;
      pair_pre(kind, kind == KIND_PP ? Cpl<T>{1, 0} : A.w2n[k], x1, x2, z1, z2);
      if (o2 != o1) buf[o2] = z2;
      buf[o1] = z1;
    }
  } else {
    for (int t = threadIdx.x; t < A.F.n * S.cols; t += nt) {
      int j, c;
      cm.split(t, j, c);
      const int o = fft_row(A.perm[j], A.F, S.s1, S.rp) + c;
      const Cpl<T> v = cx_mul(buf[o], A.t4a[j]);
      buf[o] = Cpl<T>{v.re, -v.im};  // forward = conj(inverse(conj))
    }
  }
  __syncthreads();
  fft_all<true>(buf, A.F, S.s1, cm, A.tw, nt);
  if (!pair) {
    for (int t = threadIdx.x; t < A.F.n * S.cols; t += nt) {
      int k, c;
      cm.split(t, k, c);
      const int o = fft_row(k, A.F, S.s1, S.rp) + c;
      const Cpl<T> z = buf[o];
      const Cpl<T> y = cx_mul(Cpl<T>{z.re, -z.im}, A.t4b[k]);
      buf[o] = Cpl<T>{(T)2 * y.re, (T)-2 * y.im};
    }
    __syncthreads();
  }
}

// One wavenumber's solve by one CTA of nt threads, the whole plane in shared memory: f -> u (global
// plane of this wavenumber, plane cell order).
template <typename T>
__device__ void plane_direct(const PlaneArgs<T>& O, T sg, int q, const T* __restrict__ f, T* __restrict__ u,
                             unsigned char* smem, int nt) {
  T* bt = reinterpret_cast<T*>(smem);
  T* ex = bt + O.buffers;
  T* alpha = ex + 7 * nt;
  T* num = alpha + IFACE_MAX_ENDS;
  double* work = reinterpret_cast<double*>(num + IFACE_MAX_ENDS);
  const int ncell = (int)O.ncell;
  if (threadIdx.x < 2 * IFACE_MAX_ENDS) alpha[threadIdx.x] = 0;
  size_t b0 = 0;
  for (int p = 0; p < O.np; ++p) {  // an odd number of lines: the last pair column's missing one
    const DirectArgs<T>& A = O.pc[p];
    const PlaneShape S = plane_shape(A.F, A.M, A.N, A.cls);
    if (A.cls == LINES_PAIR && (A.N & 1))
      for (int m = threadIdx.x; m < A.M; m += nt) bt[b0 + 2 * (fft_row(m, A.F, S.s1, S.rp) + S.cols - 1) + 1] = 0;
    b0 += S.buf;
  }
  for (int c = threadIdx.x; c < ncell; c += nt) {
    const unsigned o = O.celloff[c];
    bt[o & 0x7fffffffu] = neg_if(o >> 31, f[c]);
  }
  __syncthreads();
  b0 = 0;
  for (int p = 0; p < O.np; ++p) {
    const DirectArgs<T> A = O.pc[p];
    const PlaneShape S = plane_shape(A.F, A.M, A.N, A.cls);
    piece_forward(A, S, reinterpret_cast<Cpl<T>*>(bt + b0), nt);
    if (O.I.k) piece_tri<T, true>(A, S, bt + b0, sg, (T)0, ex, work, num + p, nt);
    b0 += S.buf;
  }
  if (O.I.k) {
    __syncthreads();
    iface_solve(O.I, q, work, num, alpha, nt, [&](int e, T v) {
      size_t b = 0;
      for (int p = 0; p < O.np; ++p) {
        const DirectArgs<T>& A = O.pc[p];
        const PlaneShape S = plane_shape(A.F, A.M, A.N, A.cls);
        const int ns = A.cls == LINES_PAIR ? 1 : 2;
        if (A.e0 >= 0 && e >= A.e0 && e < A.e0 + A.M) bt[b + slot_at(A, S, e - A.e0)] += v;
        if (A.e1 >= 0 && e >= A.e1 && e < A.e1 + A.M) bt[b + slot_at(A, S, e - A.e1) + (A.N - 1) * ns] += v;
        b += S.buf;
      }
    });
  }
  b0 = 0;
  for (int p = 0; p < O.np; ++p) {
    const DirectArgs<T> A = O.pc[p];
    const PlaneShape S = plane_shape(A.F, A.M, A.N, A.cls);
    piece_tri<T, false>(A, S, bt + b0, sg, alpha[p], ex, nullptr, nullptr, nt);
    piece_backward(A, S, reinterpret_cast<Cpl<T>*>(bt + b0), nt);
    b0 += S.buf;
  }
  for (int c = threadIdx.x; c < ncell; c += nt) {
    const unsigned o = O.celloff[c];
    u[c] = neg_if(o >> 31, bt[o & 0x7fffffffu]);
  }
  __syncthreads();  // the shared memory is free for the next wavenumber
}

}  // namespace
}  // namespace snac
