// The interface systems of direct solves with several pieces (direct_dev.cuh). With the pieces solved under
// Neumann faces where they meet, the jump of u across interface cell j is
//   u_b - u_a = phi_j,   A_p u = f + sum_j (-c_a phi_j at a_j, +c_b phi_j at b_j),
// so (I - Y^T R_q Z^T) phi = Y^T (end values of the solution for f): Z takes the fluxes to the spectral
// right-hand sides of the pieces' end rows, R_q holds each system's response of its end rows to its end
// rows, Y takes end values to jumps. A piece without a Dirichlet face is singular for a zero shift, and nearly
// so for a small one: R of its slot 0 then grows like 1 / shift and swamps the system (with shift -1e-8 of a
// unit box no step reduced the residual in FP64, with -1e-4 none in FP32). So where some wavenumber's shift is
// small (build_piece) that slot's system is pinned, for every wavenumber: its last unknown alpha is an unknown of
// the interface system, all others follow from it by h (1 at a zero shift) and its last row, eliminated, is the
// extra equation den alpha = num. The inverse of every system is kept with the plan, one for all wavenumbers of
// equal shift (a row of DirectPlan::d_qrow).
#include <cmath>
#include <vector>

#include "direct_dev.cuh"

namespace snac {
namespace {

// R of one system: responses of the first / last unknown to a unit right-hand side in the first / last row
// (as the solve scales them), {00, 0N, N0, NN}. Of a pinned system also {h of the first row, what a unit in the
// first row leaves in the eliminated last one, den}.
__global__ void __launch_bounds__(128) k_resp(const TriRow<double>* __restrict__ tri, const double* __restrict__ lam,
                                            const double* __restrict__ sigma, const int* __restrict__ qof,
                                            double cscale, double scale, int nq,
                                            int M, int N, int pin, double4* __restrict__ resp,
                                            double4* __restrict__ pinned) {
  const long long sys = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (sys >= (long long)nq * M) return;
  const int q = (int)(sys / M), kap = (int)(sys - (long long)q * M);
  const double tq = -fma(sigma[qof[q]], cscale, lam[kap]);
  double g = 0, d = 0, pi = 1, F = 0, inv = 0, plast = 1;
  for (int n = 0; n < N; ++n) {
    const TriRow<double> w = tri[n];
    const double s = fma(w.lo, g, w.tau + tq), den = s + w.hi;
    inv = den > 0 ? 1.0 / den : 0.0;
    d = n == 0 ? 1.0 : w.lo * d;
    if (n == N - 1 && pin && kap == 0) {
      pinned[q] = make_double4(pi, d, den, 0.0);
      inv = 0.0;
    }
    g = s * inv;
    d *= inv;
    F = fma(pi, d, F);
    plast = pi;
    pi *= w.hi * inv;
  }
  resp[sys] = make_double4(-scale * F, -scale * plast * inv, -scale * d, -scale * inv);
}

// R restricted to the cells of an end needs no product of matrices where the transform is a cosine or sine one:
// the entries of B R F depend on the difference and the sum of the two cells only, through
//   C(d) = sum_kappa h_kappa R_kappa cos(pi a_kappa d / 2M),   d < 2M
// (products of cosines or sines as sums; h: 1/2 for the first and, periodic, the last slot). One CTA per row of
// wavenumbers and piece, for every pair of its ends: 2 M^2 terms in place of k^2 M multiply-adds. Bound by the FP64 pipe
// (92 to 94 % busy); with k_build on the L of 512 x 512 x 128 cells 10.8 -> 1.0 ms.
struct CsumArgs {
  int M, kind, slots, a0, da;    // a_kappa = a0 + kappa da, kappa < slots
  int ne, u[2], ee[2];           // ends of the piece
  long long off[2][2];           // of the pair's sums within a row
  const double4* resp;           // [row][kappa]
};
__global__ void __launch_bounds__(512) k_csum(const CsumArgs A, long long stride, double* __restrict__ out) {
  extern __shared__ double cs[];  // cos(pi t / 2M), t = 0..2M
  const int M = A.M, T4 = 4 * M;
  for (int t = threadIdx.x; t <= 2 * M; t += blockDim.x) cs[t] = cospi((double)t / (2 * M));
  __syncthreads();
  const double4* R = A.resp + (size_t)blockIdx.x * M;
  double* o = out + (size_t)blockIdx.x * stride;
  for (int d = threadIdx.x; d < 2 * M; d += blockDim.x) {
    double acc[4] = {0, 0, 0, 0};
    int t = (int)((long long)A.a0 * d % T4);
    const int dt = (int)((long long)A.da * d % T4);  // (negative for the kinds with reversed slots)
    for (int k = 0; k < A.slots; ++k) {
      const bool half = A.kind != KIND_ND && A.kind != KIND_DN && (k == 0 || (A.kind == KIND_PP && 2 * k == M));
      const double c = (half ? 0.5 : 1.0) * cs[t <= 2 * M ? t : T4 - t];
      const double4 r = R[k];
      acc[0] = fma(r.x, c, acc[0]);
      acc[1] = fma(r.y, c, acc[1]);
      acc[2] = fma(r.z, c, acc[2]);
      acc[3] = fma(r.w, c, acc[3]);
      t += dt;
      t += t < 0 ? T4 : 0;
      t -= t >= T4 ? T4 : 0;
    }
    for (int a = 0; a < A.ne; ++a)
      for (int b = 0; b < A.ne; ++b) o[A.off[a][b] + d] = acc[2 * A.ee[a] + A.ee[b]];
  }
}

struct BuildArgs {
  int k, kk, E, ns, qs, nends;
  int ep[IFACE_MAX_ENDS], ee[IFACE_MAX_ENDS], eo[IFACE_MAX_ENDS + 1], sp[IFACE_MAX_ENDS];
  int em[IFACE_MAX_ENDS];                 // slots of the end's piece
  double sc[IFACE_MAX_ENDS];              // scale of the right-hand sides of a pinned piece
  const double4* pinned[IFACE_MAX_ENDS];  // of a pinned piece, [q]
  int kind[IFACE_MAX_ENDS];               // of the end's piece; -1: dense
  int co[IFACE_MAX_ENDS][IFACE_MAX_ENDS];  // cosine sums of a pair of ends within a row, -1: other piece or dense
  long long cstride;
  const double* csum;
  const IfaceCellDev* cells;
  const double4* resp[IFACE_MAX_ENDS];    // of the end's piece, [q][kappa]
  const double* Y;
  const double* Z;
};

// The transpose of K = I - Y^T R_q Z^T (KT[q][i][j] = K[j][i]), a 32 x 32 tile per CTA of 256 threads (2 x 2
// entries each); the rows and columns of the pinned pieces' unknowns beyond. Transposed, so that its inverse
// stands as the solve reads it (consecutive entries of a column of K^-1) without another copy.
constexpr int KT = 32;
__global__ void __launch_bounds__(256) k_build(const BuildArgs A, double* __restrict__ K) {
  __shared__ double ys[KT][KT + 1], ws[KT][KT + 1];
  const int q = blockIdx.z, j0 = blockIdx.y * KT, i0 = blockIdx.x * KT;
  const int tx = threadIdx.x % 16, ty = threadIdx.x / 16;
  double acc[2][2] = {{0, 0}, {0, 0}};
  for (int u = 0; u < A.nends; ++u) {  // dense transforms: products of matrices
    if (A.kind[u] >= 0) continue;
    const int M = A.em[u];
    for (int k0 = 0; k0 < M; k0 += KT) {
      for (int t = threadIdx.x; t < KT * KT; t += 256) {
        const int r = t / KT, c = t % KT;
        // ys[slot][j]
        ys[r][c] = k0 + r < M && j0 + c < A.k ? A.Y[(size_t)(A.eo[u] + k0 + r) * A.kk + j0 + c] : 0.0;
        // ws[slot][i] = sum over the ends of the same piece of R Z
        double w = 0.0;
        const int kap = k0 + c, i = i0 + r;
        if (kap < M && i < A.k) {
          const double4 R = A.resp[u][(size_t)q * M + kap];
          for (int v = 0; v < A.nends; ++v)
            if (A.ep[v] == A.ep[u]) {
              const double rr = A.ee[u] ? (A.ee[v] ? R.w : R.z) : (A.ee[v] ? R.y : R.x);
              w = fma(rr, A.Z[(size_t)i * A.E + A.eo[v] + kap], w);
            }
        }
        ws[c][r] = w;
      }
      __syncthreads();
#pragma unroll 8
      for (int e = 0; e < KT; ++e) {
        const double a0 = ys[e][tx], a1 = ys[e][tx + 16], b0 = ws[e][ty], b1 = ws[e][ty + 16];
        acc[0][0] = fma(a0, b0, acc[0][0]);
        acc[0][1] = fma(a0, b1, acc[0][1]);
        acc[1][0] = fma(a1, b0, acc[1][0]);
        acc[1][1] = fma(a1, b1, acc[1][1]);
      }
      __syncthreads();
    }
  }
  for (int a = 0; a < 2; ++a)
    for (int b = 0; b < 2; ++b) {
      const int j = j0 + tx + 16 * a, i = i0 + ty + 16 * b;
      if (j >= A.kk || i >= A.kk) continue;
      double v = (j == i ? 1.0 : 0.0) - acc[a][b];
      if (j < A.k && i < A.k) {
        const IfaceCellDev cj = A.cells[j], ci = A.cells[i];
        for (int x = 0; x < 2; ++x)
          for (int y = 0; y < 2; ++y) {
            const int o = A.co[cj.u[x]][ci.u[y]];
            if (o < 0) continue;
            const double* C = A.csum + (size_t)q * A.cstride + o;
            const int kind = A.kind[cj.u[x]], mj = cj.m[x], mi = ci.m[y];
            const double c0 = C[mj > mi ? mj - mi : mi - mj];
            const double g = kind == KIND_PP ? 4.0 * c0
                             : kind == KIND_NN || kind == KIND_ND ? 2.0 * (c0 + C[mj + mi + 1]) : 2.0 * (c0 - C[mj + mi + 1]);
            v = fma(x == 0 ? g : -g, ci.z[y], v);  // - Y (R Z): Y is -1 below, +1 above
          }
      } else {
        v = j == i ? 1.0 : 0.0;
        if (!(q == A.qs && j == A.kk - 1)) {  // (the last equation of a singular problem is implied: alpha = 0)
          const int a = (j < A.k ? i : j) - A.k, p = A.sp[a];
          const double4 R = A.pinned[a][q];
          v = j == i ? R.z : 0.0;
          if (j < A.k || i < A.k)
            for (int u = 0; u < A.nends; ++u)
              if (A.ep[u] == p)
                v += j < A.k ? -A.Y[(size_t)A.eo[u] * A.kk + j] * (A.ee[u] ? 1.0 : R.x)
                             : A.sc[a] * A.Z[(size_t)i * A.E + A.eo[u]] * (A.ee[u] ? 1.0 : R.y);
        }
      }
      K[((size_t)q * A.kk + i) * A.kk + j] = v;
    }
}

// In-place Gauss-Jordan inverse of every K, one CTA each. No pivoting: K is the identity plus a product
// of positive operators, and the pinned unknowns come last. Bound by the FP64 pipe (128 systems of 256: 5.4 ms, 91 %
// busy) or, for smaller systems, by the latency of a step: 1024 threads from 64 unknowns on (96 systems of 160 with
// 256 threads 5.7 ms, 49 with 1024 2.1 ms).
__global__ void __launch_bounds__(1024) k_invert(double* __restrict__ Kq, int n) {
  extern __shared__ double sh[];
  double* rp = sh;        // pivot row / pivot
  double* cp = sh + n;    // pivot column
  double* K = Kq + (size_t)blockIdx.x * n * n;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  for (int p = 0; p < n; ++p) {
    const double piv = 1.0 / K[(size_t)p * n + p];
    for (int j = threadIdx.x; j < n; j += blockDim.x) {
      rp[j] = j == p ? piv : K[(size_t)p * n + j] * piv;
      cp[j] = K[(size_t)j * n + p];
    }
    __syncthreads();
    for (int i = warp; i < n; i += nw) {
      double* row = K + (size_t)i * n;
      const double c = cp[i];
      for (int j = lane; j < n; j += 32)
        row[j] = i == p ? rp[j] : (j == p ? -c * piv : fma(-c, rp[j], row[j]));
    }
    __syncthreads();
  }
}

constexpr int INT = 1024;

// One wavenumber per CTA: fluxes from the end values, added to the spectral right-hand sides. Bound by
// reading Y, Z (shared by all wavenumbers, L2) and the kept inverse.
template <typename T>
__global__ void __launch_bounds__(INT) k_iface(const IfaceArgs<T> I, long long ncell, T* __restrict__ x) {
  extern __shared__ __align__(16) unsigned char raw[];
  double* work = reinterpret_cast<double*>(raw);
  const int q = blockIdx.x;
  for (int e = threadIdx.x; e < I.E; e += INT) work[e] = (double)I.ends[(size_t)q * I.E + e];
  __syncthreads();
  T* xq = x + (long long)q * ncell;
  iface_solve(I, q, work, I.num + q * IFACE_MAX_ENDS, I.alpha + q * IFACE_MAX_ENDS, INT, [&](int e, T v) {
    int u = 0;
    while (u + 1 < I.nends && e >= I.eo[u + 1]) ++u;
    xq[I.row[u] + e - I.eo[u]] += v;
  });
}

template <typename T>
cudaError_t iface_t(snac_plan* P, cudaStream_t s) {
  const IfaceArgs<T> I = iface_args<T>(P);
  const size_t smem = iface_doubles(I.E, I.kk, INT) * sizeof(double);
  LaunchScope ls(P, K_IFACE, P->nz * (8.0 * I.kk * I.kk + 3.0 * sizeof(T) * I.E),
                 2.0 * P->nz * ((double)I.kk * I.kk + 2.0 * I.k * I.E), s);
  cudaFuncSetAttribute(k_iface<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, 128 * 1024);
  k_iface<T><<<P->nz, INT, smem, s>>>(I, P->lev[0].ncell, (T*)P->lev[0].d_u);
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_iface(snac_plan* P, cudaStream_t s) {
  return P->precision == SNAC_FP64 ? iface_t<double>(P, s) : iface_t<float>(P, s);
}

cudaError_t setup_iface(snac_plan* P, const int* d_qof, int rows, int qs_row, cudaStream_t s) {
  DirectPlan& D = P->direct;
  IfaceTab& I = D.it;
  const bool f64 = P->precision == SNAC_FP64;
  // temporaries in stream order: cudaFree would wait for every other stream of the device
  std::vector<void*> tmp;
  cudaError_t e = cudaSuccess;
  auto get = [&](size_t bytes) -> void* {
    void* p = nullptr;
    if (e == cudaSuccess) e = cudaMallocAsync(&p, bytes, s);
    if (p) tmp.push_back(p);
    return p;
  };
  BuildArgs A{};
  A.k = I.k;
  A.kk = I.kk;
  A.E = I.E;
  A.ns = I.ns;
  A.qs = qs_row;
  A.nends = I.nends;
  for (int a = 0; a < I.ns; ++a) A.sp[a] = I.sp[a];
  double* dZ = (double*)get(I.Zh.size() * sizeof(double));
  if (e == cudaSuccess) e = cudaMemcpyAsync(dZ, I.Zh.data(), I.Zh.size() * sizeof(double), cudaMemcpyHostToDevice, s);
  A.Y = I.d_Y;
  A.Z = dZ;
  std::vector<double4*> resp(D.pc.size(), nullptr), pinned(D.pc.size(), nullptr);
  for (size_t p = 0; p < D.pc.size(); ++p) {
    const DirectTab& d = D.pc[p];
    resp[p] = (double4*)get((size_t)rows * d.M * sizeof(double4));
    if (d.pin) pinned[p] = (double4*)get((size_t)rows * sizeof(double4));
    if (e != cudaSuccess) break;
    const TriRow<double>* tri = (const TriRow<double>*)(f64 ? d.d_tri : (void*)d.d_tri64);
    const double* lam = f64 ? (const double*)d.d_lam : d.d_lam64;
    const long long sys = (long long)rows * d.M;
    k_resp<<<(unsigned)((sys + 127) / 128), 128, 0, s>>>(tri, lam, P->d_sigma64, d_qof, d.cscale, d.cscale / d.theta, rows,
                                                        d.M, d.N, d.pin, resp[p], pinned[p]);
    e = cudaGetLastError();
  }
  for (int u = 0; u <= I.nends; ++u) A.eo[u] = I.eo[u];
  for (int u = 0; u < I.nends; ++u) {
    const DirectTab& d = D.pc[I.ep[u]];
    A.ep[u] = I.ep[u];
    A.ee[u] = I.ee[u];
    A.em[u] = d.M;
    A.resp[u] = resp[I.ep[u]];
  }
  // cosine sums of the pieces with a cosine or sine transform
  for (auto& row : A.co)
    for (int& o : row) o = -1;
  std::vector<CsumArgs> cs;
  for (size_t p = 0; p < D.pc.size(); ++p) {
    const DirectTab& d = D.pc[p];
    CsumArgs c{};
    for (int u = 0; u < I.nends; ++u) {
      if (I.ep[u] != (int)p) continue;
      A.kind[u] = d.cls == LINES_DENSE ? -1 : d.kind;
      c.u[c.ne] = u;
      c.ee[c.ne++] = I.ee[u];
    }
    if (d.cls == LINES_DENSE || c.ne == 0) continue;
    c.M = d.M;
    c.kind = d.kind;
    c.slots = d.kind == KIND_PP ? d.M / 2 + 1 : d.M;
    c.a0 = d.kind == KIND_DD ? 2 * d.M : d.kind == KIND_DN ? 2 * d.M - 1 : d.kind == KIND_ND ? 1 : 0;
    c.da = d.kind == KIND_PP ? 4 : d.kind == KIND_DD || d.kind == KIND_DN ? -2 : 2;
    c.resp = resp[p];
    for (int a = 0; a < c.ne; ++a)
      for (int b = 0; b < c.ne; ++b) {
        A.co[c.u[a]][c.u[b]] = (int)A.cstride;
        c.off[a][b] = A.cstride;
        A.cstride += 2 * d.M;
      }
    cs.push_back(c);
  }
  double* csum = (double*)get((size_t)rows * A.cstride * sizeof(double));
  IfaceCellDev* cells = (IfaceCellDev*)get(I.cells.size() * sizeof(IfaceCellDev));
  if (e == cudaSuccess)
    e = cudaMemcpyAsync(cells, I.cells.data(), I.cells.size() * sizeof(IfaceCellDev), cudaMemcpyHostToDevice, s);
  A.csum = csum;
  A.cells = cells;
  for (const CsumArgs& c : cs) {
    if (e != cudaSuccess) break;
    cudaFuncSetAttribute(k_csum, cudaFuncAttributeMaxDynamicSharedMemorySize, 80 * 1024);  // (M <= MAX_NZ)
    k_csum<<<rows, 512, (2 * (size_t)c.M + 1) * sizeof(double), s>>>(c, A.cstride, csum);
    e = cudaGetLastError();
  }
  for (int a = 0; a < I.ns; ++a) {
    A.sc[a] = D.pc[I.sp[a]].cscale / D.pc[I.sp[a]].theta;
    A.pinned[a] = pinned[I.sp[a]];
  }
  if (e == cudaSuccess) {
    const unsigned t = (unsigned)((I.kk + KT - 1) / KT);
    k_build<<<dim3(t, t, (unsigned)rows), 256, 0, s>>>(A, I.d_KT);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) {
    const size_t smem = 2 * (size_t)I.kk * sizeof(double);
    k_invert<<<rows, I.kk >= 64 ? 1024 : 256, smem, s>>>(I.d_KT, I.kk);
    e = cudaGetLastError();
  }
  for (void* p : tmp) {
    const cudaError_t ef = cudaFreeAsync(p, s);
    if (e == cudaSuccess) e = ef;
  }
  const cudaError_t es = cudaStreamSynchronize(s);
  if (e == cudaSuccess) e = es;
  std::vector<double>().swap(I.Zh);
  std::vector<IfaceCellDev>().swap(I.cells);
  return e;
}

}  // namespace snac
