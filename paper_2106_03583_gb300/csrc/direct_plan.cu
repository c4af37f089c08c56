// Plan creation for direct solves of the reduced equations (direct_dev.cuh): which layouts allow them, the
// pieces, and their tables.
//
// Blocks connected along the transformed axis form chains; chains stacked on one another along the other
// axis with every face connected form a piece: a rectangle with one tensor grid. A layout of one piece (any
// assembled rectangle) separates as it stands. Several pieces (L and T shapes, a channel with a side
// branch) meet along parts of their first and last rows: each piece is solved with a Neumann condition
// there, and the fluxes through the shared faces follow from a dense system per wavenumber (kern_iface.cu).
#include <algorithm>
#include <atomic>
#include <cmath>
#include <map>
#include <new>
#include <thread>
#include <vector>

#include "direct_dev.cuh"

namespace snac {
void set_error(const std::string& s);

// Passes of an in-place FFT of n points: the factors 2 spread evenly over the fewest passes of at most
// max_log2 each, then 7, 5, 3. False if another prime divides n.
bool fft_tab(int n, int max_log2, FftTab& F) {
  F = FftTab{};
  F.n = n;
  int twos = 0, rest = n;
  while (rest % 2 == 0) rest /= 2, ++twos;
  std::vector<int> rad;
  for (int left = twos, np = (twos + max_log2 - 1) / max_log2; np > 0; --np) {
    const int b = (left + np - 1) / np;
    rad.push_back(1 << b);
    left -= b;
  }
  for (int p : {7, 5, 3})
    while (rest % p == 0) rest /= p, rad.push_back(p);
  if (rest != 1 || rad.size() > FFT_MAX_PASS) return false;
  if (rad.empty()) rad.push_back(1);
  F.np = n == 1 ? 0 : (int)rad.size();
  F.l1 = n / rad[0];
  F.l1r = recip16(F.l1);
  int span = n;
  for (int k = 0; k < F.np; ++k) {
    F.rad[k] = rad[k];
    F.span[k] = span;
    F.lr[k] = recip16(span / rad[k]);
    F.pr[k] = recip16(std::max(F.l1 / span, 1));
    span /= rad[k];
  }
  return true;
}

// Row of every frequency after the forward passes (digit-reversed order).
std::vector<int> fft_perm(const FftTab& F) {
  std::vector<int> perm(F.n);
  for (int k = 0; k < F.n; ++k) {
    int q = k, p = 0;
    for (int s = 0; s < F.np; ++s) {
      p += (q % F.rad[s]) * (F.span[s] / F.rad[s]);
      q /= F.rad[s];
    }
    perm[k] = p;
  }
  return perm;
}

namespace {

// Boundary pair of an axis from its two outer face kinds.
int pair_kind(int lo, int hi) {
  if (lo == SNAC_BC_PERIODIC) return KIND_PP;
  if (lo == SNAC_BC_NEUMANN) return hi == SNAC_BC_NEUMANN ? KIND_NN : KIND_ND;
  return hi == SNAC_BC_NEUMANN ? KIND_DN : KIND_DD;
}

struct Chain {
  std::vector<int> blk;
  bool ring = false;
};

// A piece while it is being described: its chains from the first row of blocks to the last.
struct Piece {
  std::vector<Chain> rows;
  int kind = 0;
  int side[2] = {0, 0};        // face kind of the first / last row (SNAC_BC_NEUMANN where it has interface cells)
  bool iface[2] = {false, false};
};

struct IfaceCell {
  int pa, ma, pb, mb;  // last row of piece pa, first row of piece pb
  double ca, cb;       // their couplings
};

struct Layout {
  int axis = 0;  // transformed axis
  std::vector<Piece> pc;
  std::vector<IfaceCell> cells;
};

// The pieces of the layout for a transformed axis; false if it does not fit the scheme.
bool pieces_along(const snac_plan* P, const std::vector<FaceKinds>& faces, int t, Layout& out) {
  const HostLevel& l0 = P->lev[0];
  const std::vector<BlockDev>& B = l0.blk;
  const int nb = (int)B.size(), tl = 2 * t, th = 2 * t + 1, nl = 2 * (1 - t), nh = 2 * (1 - t) + 1;
  out = Layout{};
  out.axis = t;
  std::vector<Chain> ch;
  std::vector<int> of(nb, -1), at(nb, -1);
  auto add = [&](int b0, bool ring) {
    Chain c;
    c.ring = ring;
    for (int b = b0; b >= 0 && of[b] < 0; b = B[b].nbr[th]) {
      of[b] = (int)ch.size();
      at[b] = (int)c.blk.size();
      c.blk.push_back(b);
    }
    ch.push_back(c);
  };
  for (int b = 0; b < nb; ++b)
    if (B[b].nbr[tl] < 0) add(b, false);
  for (int b = 0; b < nb; ++b)
    if (of[b] < 0) add(b, true);
  // the chain above, where every face matches
  const int nc = (int)ch.size();
  std::vector<int> up(nc, -1), down(nc, -1);
  for (int c = 0; c < nc; ++c) {
    const int b0 = B[ch[c].blk[0]].nbr[nh];
    if (b0 < 0 || of[b0] == c) continue;
    const int d = of[b0];
    const int n = (int)ch[c].blk.size();
    bool ok = (int)ch[d].blk.size() == n && ch[d].ring == ch[c].ring && (ch[c].ring || at[b0] == 0);
    for (int i = 0; i < n && ok; ++i) ok = B[ch[c].blk[i]].nbr[nh] == ch[d].blk[(at[b0] + i) % n];
    const FaceKinds &f0 = faces[ch[c].blk[0]], &f1 = faces[ch[c].blk.back()];
    const FaceKinds &g0 = faces[ch[d].blk[0]], &g1 = faces[ch[d].blk.back()];
    ok = ok && (ch[c].ring || (f0.k[tl] == g0.k[tl] && f1.k[th] == g1.k[th]));
    if (ok) up[c] = d, down[d] = c;
  }
  std::vector<int> piece_of(nc, -1);
  for (int c = 0; c < nc; ++c) {
    if (down[c] >= 0) continue;
    Piece p;
    for (int d = c; d >= 0; d = up[d]) {
      Chain row = ch[d];
      if (row.ring && !p.rows.empty()) {  // a ring starts wherever it was met: start above the first block
        const int b0 = B[p.rows.back().blk[0]].nbr[nh];
        std::rotate(row.blk.begin(), std::find(row.blk.begin(), row.blk.end(), b0), row.blk.end());
      }
      piece_of[d] = (int)out.pc.size();
      p.rows.push_back(row);
    }
    const Chain& r0 = p.rows[0];
    p.kind = r0.ring ? KIND_PP : pair_kind(faces[r0.blk[0]].k[tl], faces[r0.blk.back()].k[th]);
    out.pc.push_back(p);
  }
  for (int c = 0; c < nc; ++c)
    if (piece_of[c] < 0) return false;  // stacked in a circle: periodic along the tridiagonal axis
  // position of every block along its piece's transformed axis
  std::vector<int> m0(nb, 0), pof(nb, 0);
  auto ext = [&](int b, int a) { return a == 0 ? B[b].nx : B[b].ny; };
  for (size_t p = 0; p < out.pc.size(); ++p)
    for (const Chain& r : out.pc[p].rows) {
      int m = 0;
      for (int b : r.blk) {
        m0[b] = m;
        pof[b] = (int)p;
        m += ext(b, t);
      }
    }
  for (size_t p = 0; p < out.pc.size(); ++p)
    for (int e = 0; e < 2; ++e) {
      Piece& pc = out.pc[p];
      const Chain& r = e == 0 ? pc.rows.front() : pc.rows.back();
      const int f = e == 0 ? nl : nh;
      int wall = -1, links = 0;
      for (int b : r.blk) {
        if (B[b].nbr[f] >= 0) {
          ++links;
          if (pof[B[b].nbr[f]] == (int)p) return false;  // the piece meets itself
          continue;
        }
        if (wall >= 0 && wall != faces[b].k[f]) return false;
        wall = faces[b].k[f];
      }
      if (links && wall >= 0 && wall != SNAC_BC_NEUMANN) return false;  // (a Dirichlet wall beside an interface)
      pc.iface[e] = links > 0;
      pc.side[e] = links ? (int)SNAC_BC_NEUMANN : wall;
      if (e == 0 || !links) continue;
      for (int b : r.blk) {
        const int c = B[b].nbr[f];
        if (c < 0) continue;
        const Coef<double>*ka, *kb;
        if (t == 0) {
          ka = &l0.cy[B[b].yo + B[b].ny - 1];
          kb = &l0.cy[B[c].yo];
        } else {
          ka = &l0.cx[B[b].xo + B[b].nx - 1];
          kb = &l0.cx[B[c].xo];
        }
        for (int i = 0; i < ext(b, t); ++i)
          out.cells.push_back({(int)p, m0[b] + i, pof[c], m0[c] + i, ka->hi, kb->lo});
      }
    }
  return true;
}

// Widths of a piece along an axis: the blocks of its first row (transformed axis) or first column.
std::vector<double> piece_widths(const snac_plan* P, const Piece& p, int axis, bool transformed) {
  const HostLevel& l0 = P->lev[0];
  std::vector<double> w;
  auto put = [&](int b) {
    const BlockDev& d = l0.blk[b];
    if (axis == 0)
      for (int i = 0; i < d.nx; ++i) w.push_back(l0.cx[d.xo + i].w);
    else
      for (int j = 0; j < d.ny; ++j) w.push_back(l0.cy[d.yo + j].w);
  };
  if (transformed)
    for (int b : p.rows[0].blk) put(b);
  else
    for (const Chain& r : p.rows) put(r.blk[0]);
  return w;
}

// Rotations of rows k, k + 1 for k = lo .. lo + length - 1: (u, v) -> (c u + s v, c v - s u).
struct Sweep {
  int lo, length;
  size_t first;  // of their cosines and sines
};

// The sweeps in order on the identity's columns i0 .. i0 + W - 1, into Z (n x n). A row between two rotations stays
// in registers, and W columns of 384 rows in the first-level cache.
constexpr int EIG_W = 16;
void rotate_columns(const std::vector<Sweep>& sw, const std::vector<double>& cs, int n, int i0, double* Z) {
  constexpr int W = EIG_W;
  std::vector<double> z((size_t)n * W, 0.0);
  const int w = std::min(W, n - i0);
  for (int i = 0; i < w; ++i) z[(size_t)(i0 + i) * W + i] = 1.0;
  for (const Sweep& s : sw) {
    double u[W];
    double* row = &z[(size_t)s.lo * W];
    const double* r = &cs[s.first];
    for (int i = 0; i < W; ++i) u[i] = row[i];
    for (int k = 0; k < s.length; ++k, row += W, r += 2)
      for (int i = 0; i < W; ++i) {
        const double v = row[W + i];
        row[i] = r[0] * u[i] + r[1] * v;
        u[i] = r[0] * v - r[1] * u[i];
      }
    for (int i = 0; i < W; ++i) row[i] = u[i];
  }
  for (int k = 0; k < n; ++k)
    for (int i = 0; i < w; ++i) Z[(size_t)k * n + i0 + i] = z[(size_t)k * W + i];
}

// Eigenvalues (into d) and orthonormal eigenvectors (rows of Z) of a symmetric tridiagonal matrix with
// diagonal d and off-diagonal e (e[i] couples i and i + 1): shifted QR steps by Givens rotations chased down
// the unreduced block (Wilkinson's shift). False if the block of one eigenvalue takes more than 60 steps. The
// rotations, about 1.2 n^2, are applied to blocks of columns afterwards, by a few threads.
bool tridiag_eigen(std::vector<double>& d, std::vector<double> e, std::vector<double>& Z) {
  const int n = (int)d.size();
  std::vector<Sweep> sw;
  std::vector<double> cs;
  auto small = [&](int i) { return std::fabs(e[i]) <= 1.1e-16 * (std::fabs(d[i]) + std::fabs(d[i + 1])); };
  int steps = 0;
  for (int hi = n - 1; hi > 0;) {
    if (small(hi - 1)) {
      e[--hi] = 0.0;
      steps = 0;
      continue;
    }
    if (++steps > 60) return false;
    int lo = hi - 1;
    while (lo > 0 && !small(lo - 1)) --lo;
    // the eigenvalue of the trailing 2 x 2 block closer to its last entry
    const double h = 0.5 * (d[hi - 1] - d[hi]), b = e[hi - 1];
    const double mu = d[hi] - b * b / (h + std::copysign(std::hypot(h, b), h));
    double x = d[lo] - mu, z = e[lo];
    sw.push_back({lo, hi - lo, cs.size()});
    for (int k = lo; k < hi; ++k) {
      // rotate rows and columns k, k + 1 so that (x, z) becomes (r, 0)
      const double r = std::hypot(x, z), c = r > 0.0 ? x / r : 1.0, s = r > 0.0 ? z / r : 0.0;
      if (k > lo) e[k - 1] = r;
      const double d0 = d[k], d1 = d[k + 1], ek = e[k];
      d[k] = c * c * d0 + 2.0 * c * s * ek + s * s * d1;
      d[k + 1] = s * s * d0 - 2.0 * c * s * ek + c * c * d1;
      e[k] = c * s * (d1 - d0) + (c * c - s * s) * ek;
      if (k + 1 < hi) {
        x = e[k];
        z = s * e[k + 1];
        e[k + 1] *= c;
      }
      cs.push_back(c);
      cs.push_back(s);
    }
  }
  Z.resize((size_t)n * n);
  const int blocks = (n + EIG_W - 1) / EIG_W;
  std::atomic<int> next{0};
  std::atomic<bool> failed{false};
  auto work = [&] {
    try {
      for (int b; (b = next.fetch_add(1)) < blocks;) rotate_columns(sw, cs, n, b * EIG_W, Z.data());
    } catch (...) {
      failed = true;
    }
  };
  std::vector<std::thread> th;
  const int want = std::min({7, blocks / 2, (int)std::thread::hardware_concurrency() - 1});
  try {
    for (int t = 0; t < want; ++t) th.emplace_back(work);
  } catch (...) {  // no more threads: the ones there are do
  }
  work();
  for (std::thread& t : th) t.join();
  if (failed) throw std::bad_alloc();
  return true;
}

bool uniform(const std::vector<double>& w) {
  for (double v : w)
    if (std::fabs(v - w[0]) > 1e-12 * w[0]) return false;
  return true;
}

// Whether a piece's lines take the FFT: a uniform axis of even length whose half (DCT-IV kinds) or whole
// has no prime factor above 7.
bool fft_piece(const Piece& p, const std::vector<double>& w) {
  const int m = (int)w.size();
  FftTab F;
  const bool four = p.kind == KIND_ND || p.kind == KIND_DN;
  return m % 2 == 0 && m >= 4 && m <= MAX_NZ && uniform(w) && fft_tab(four ? m / 2 : m, 4, F);
}

// Operations per plane cell of a layout's transforms and interfaces; negative if some piece can't be
// transformed. Dense transforms (2 M FMA per cell and solve) only for planes of several passes, and where they
// beat the V-cycles they replace, which take the longer the more the plane is stretched: measured on M x M x 160
// cells, stretched mildly both ways, FP64 3.2 -> 1.9 ms at M = 128, 5.9 -> 5.2 at 192, but 9.9 -> 11.3 at 256:
// up to 200 cells on average over the plane; mixed 2.1 -> 0.7, 2.9 -> 1.2, 4.4 -> 3.2 and 8.3 -> 7.7 at 384: up
// to there (the eigenvectors, O(M^3) on the host, take 0.02 s of plan creation). 336 x 192 x 150 mixed 6.1 -> 1.6
// to 2.1 ms; three rectangles of 64 to 128 cells by 192, FP64, 3.6 -> 2.0 ms.
double layout_cost(const snac_plan* P, const Layout& L) {
  const bool f64 = P->precision == SNAC_FP64;
  double ops = 0.0, cells = 0.0, dense = 0.0, ends = 0.0;
  for (const Piece& p : L.pc) {
    const std::vector<double> w = piece_widths(P, p, L.axis, true);
    const double m = (double)w.size(), n = (double)piece_widths(P, p, 1 - L.axis, false).size();
    if (n < 2 || n > 65535) return -1.0;
    cells += m * n;
    for (int e = 0; e < 2; ++e) ends += p.iface[e] ? m : 0.0;
    if (fft_piece(p, w)) {
      ops += 30.0 * m * n;
      continue;
    }
    if (P->onchip || p.kind == KIND_PP || m < 4 || m > 384) return -1.0;
    dense += m * m * n;
  }
  if (f64 && dense > 200.0 * cells) return -1.0;
  const double k = (double)L.cells.size();
  return (ops + 2.0 * dense + k * (k + 2.0 * ends)) / cells;
}

std::vector<float> to_float(const std::vector<double>& v) { return std::vector<float>(v.begin(), v.end()); }

// A table in the plan's inner type.
int up_inner(snac_plan* P, void** d, const std::vector<double>& v) {
  if (P->precision == SNAC_FP64) return plan_upload(P, d, v.data(), v.size() * sizeof(double));
  const std::vector<float> f = to_float(v);
  return plan_upload(P, d, f.data(), f.size() * sizeof(float));
}
template <typename V>
int up_vec(snac_plan* P, V** d, const std::vector<V>& v) {
  return plan_upload(P, reinterpret_cast<void**>(d), v.data(), v.size() * sizeof(V));
}

// The shift of every wavenumber of the problem (a plan may hold a range of them only).
std::vector<double> all_shifts(const snac_plan* P) {
  const double iz2 = 1.0 / (P->dz * P->dz);
  std::vector<double> sigma(P->nzt);
  for (int q = 0; q < P->nzt; ++q) sigma[q] = mode_lambda(P->kind, P->nzt, q) * iz2 + P->shift;
  return sigma;
}

// The layout has no direct solve after all: the plan keeps its V-cycles.
constexpr int NOT_DIRECT = 1;

int build_piece(snac_plan* P, const Piece& p, int ax, int soff, DirectTab& D) {
  const HostLevel& l0 = P->lev[0];
  const bool f64 = P->precision == SNAC_FP64;
  const std::vector<double> wm = piece_widths(P, p, ax, true);
  D.M = (int)wm.size();
  D.N = (int)piece_widths(P, p, 1 - ax, false).size();
  D.kind = p.kind;
  D.cls = !fft_piece(p, wm) ? LINES_DENSE : p.kind == KIND_ND || p.kind == KIND_DN ? LINES_DCT4 : LINES_PAIR;
  D.xl = ax == 0 ? 1 : 0;
  D.soff = soff;
  if (D.cls == LINES_DENSE) fft_tab(2, 1, D.fft);  // (not used)
  else fft_tab(D.cls == LINES_PAIR ? D.M : D.M / 2, f64 ? 3 : 4, D.fft);
  const int nf = D.fft.n, M = D.M, N = D.N;
  D.theta = D.cls == LINES_DENSE ? 1.0 : 2.0 * M;
  D.w2n = nf;
  D.t4a = D.w2n + M + 1;
  D.t4b = D.t4a + M / 2;
  std::vector<double> tw(2 * (size_t)(D.t4b + M / 2));
  auto put = [&](int k, double ang) {
    tw[2 * k] = std::cos(ang);
    tw[2 * k + 1] = std::sin(ang);
  };
  for (int k = 0; k < nf; ++k) put(k, -2.0 * M_PI * k / nf);
  for (int k = 0; k <= M; ++k) put(D.w2n + k, -M_PI * k / (2.0 * M));
  for (int k = 0; k < M / 2; ++k) put(D.t4a + k, -M_PI * (4.0 * k + 1.0) / (4.0 * M));
  for (int k = 0; k < M / 2; ++k) put(D.t4b + k, -M_PI * k / (double)M);
  const std::vector<int> perm = fft_perm(D.fft);
  // eigenvalues of the slots and the tridiagonal rows, scaled by a power of two to couplings of about 1 (cell
  // widths in any unit: their squares may lie near the ends of the range)
  double h = 0.0;
  for (double v : wm) h += v;
  h /= M;
  std::vector<Coef<double>> ct;
  for (const Chain& r : p.rows) {
    const BlockDev& d = l0.blk[r.blk[0]];
    if (ax == 0) ct.insert(ct.end(), l0.cy.begin() + d.yo, l0.cy.begin() + d.yo + d.ny);
    else ct.insert(ct.end(), l0.cx.begin() + d.xo, l0.cx.begin() + d.xo + d.nx);
  }
  ct.front().lo = 0.0;  // (an interface is a Neumann face of the piece)
  ct.back().hi = 0.0;
  std::vector<Coef<double>> cm;
  if (D.cls == LINES_DENSE)
    for (int b : p.rows[0].blk) {
      const BlockDev& d = l0.blk[b];
      if (ax == 0) cm.insert(cm.end(), l0.cx.begin() + d.xo, l0.cx.begin() + d.xo + d.nx);
      else cm.insert(cm.end(), l0.cy.begin() + d.yo, l0.cy.begin() + d.yo + d.ny);
    }
  double big = D.cls == LINES_DENSE ? 0.0 : 4.0 / (h * h);
  for (const Coef<double>& c : cm) big = std::max(big, -2.0 * c.d);
  bool finite = true;
  for (const Coef<double>& c : ct) {
    big = std::max(big, c.lo + c.hi);
    finite = finite && std::isfinite(c.d);
  }
  if (!finite || !std::isfinite(big)) return NOT_DIRECT;
  int ex = 0;
  std::frexp(big, &ex);
  D.cscale = std::ldexp(1.0, -ex);
  // dense: A = W^-1/2 Q Lam Q^T W^1/2 along the axis, F = Q^T W^1/2, B = W^-1/2 Q, smallest |lambda| first
  std::vector<double> ev;
  if (D.cls == LINES_DENSE) {
    std::vector<double> dd(M), ee(M, 0.0), Z;
    for (int m = 0; m < M; ++m) {
      dd[m] = D.cscale * cm[m].d;
      if (m + 1 < M) ee[m] = std::sqrt((D.cscale * cm[m].hi) * (D.cscale * cm[m + 1].lo));
    }
    if (!tridiag_eigen(dd, ee, Z)) return NOT_DIRECT;
    std::vector<int> order(M);
    for (int k = 0; k < M; ++k) order[k] = k;
    std::sort(order.begin(), order.end(), [&](int a, int b) { return dd[a] > dd[b]; });
    D.F.resize((size_t)M * M);
    D.B.resize((size_t)M * M);
    std::vector<double> ft((size_t)M * M), bt((size_t)M * M);
    ev.resize(M);
    for (int k = 0; k < M; ++k) {
      ev[k] = std::min(0.0, dd[order[k]]);
      if (k == 0 && p.kind == KIND_NN) ev[k] = 0.0;
      for (int m = 0; m < M; ++m) {
        const double q = Z[(size_t)order[k] * M + m], r = std::sqrt(wm[m]);
        D.F[(size_t)k * M + m] = ft[(size_t)m * M + k] = q * r;
        D.B[(size_t)m * M + k] = bt[(size_t)k * M + m] = q / r;
      }
    }
    int se;
    if ((se = up_inner(P, &D.d_F, ft)) || (se = up_inner(P, &D.d_B, bt))) return se;
  }
  D.lam.resize(M);
  for (int k = 0; k < M; ++k)
    D.lam[k] = !ev.empty() ? ev[k] : D.cscale * mode_lambda(p.kind, M, p.kind == KIND_DD || p.kind == KIND_DN ? M - 1 - k : k) / (h * h);
  std::vector<double> tri(4 * (size_t)N);
  for (int n = 0; n < N; ++n) {
    const Coef<double>& c = ct[n];
    double tau = 0.0;
    if (n == 0 && p.side[0] == SNAC_BC_DIRICHLET) tau += 2.0 / (c.w * c.w);
    if (n == N - 1 && p.side[1] == SNAC_BC_DIRICHLET) tau += 2.0 / (c.w * c.w);
    tri[4 * n] = D.cscale * c.lo;
    tri[4 * n + 1] = D.cscale * c.hi;
    tri[4 * n + 2] = D.cscale * tau;
    tri[4 * n + 3] = c.hi > 0.0 ? c.lo / c.hi : 0.0;
  }
  // slot 0 of an all-Neumann or periodic piece is nearly singular for shifts well below the next slot's eigenvalue:
  // not pinned, a mixed L of 256 x 160 cells took a third step at a tenth of it, a fourth at a thousandth. Above a
  // quarter its response is like theirs, and the interface systems stay one unknown smaller
  D.pin = (p.iface[0] || p.iface[1]) && (p.kind == KIND_PP || p.kind == KIND_NN) && p.side[0] != SNAC_BC_DIRICHLET &&
          p.side[1] != SNAC_BC_DIRICHLET;
  if (D.pin) {
    double next = -INFINITY, least = INFINITY;
    for (int k = 1; k < M; ++k) next = std::max(next, D.lam[k]);
    for (double s : all_shifts(P)) least = std::min(least, -s * D.cscale);
    D.pin = least < -0.25 * next;
  }
  // where the lines live: plane offset of (m, n) = base[n nbm + mblk[m]] + m mstr[n]
  const int gm = (int)p.rows[0].blk.size();
  std::vector<int>&mblk = D.mblk, &base = D.base, &mstr = D.mstr;
  mblk.resize(M), base.resize((size_t)N * gm), mstr.resize(N);
  bool vec = l0.ncell % 2 == 0 && (ax == 0 || N % 2 == 0);
  int n0 = 0;
  for (const Chain& r : p.rows) {
    int m0 = 0;
    for (int i = 0; i < gm; ++i) {
      const BlockDev& d = l0.blk[r.blk[i]];
      const int em = ax == 0 ? d.nx : d.ny, en = ax == 0 ? d.ny : d.nx;
      // pairs are two cells of a line (x lines), or the same cell of two adjacent lines (the first even)
      vec = vec && d.off % 2 == 0 && d.nx % 2 == 0 && (ax == 0 ? m0 : n0) % 2 == 0;
      for (int m = m0; m < m0 + em; ++m) mblk[m] = i;
      for (int n = n0; n < n0 + en; ++n) {
        mstr[n] = ax == 0 ? 1 : d.nx;
        const long long c = ax == 0 ? d.off + (long long)(n - n0) * d.nx : d.off + (n - n0);
        base[(size_t)n * gm + i] = (int)(c - (long long)m0 * mstr[n]);
      }
      m0 += em;
    }
    n0 += ax == 0 ? l0.blk[r.blk[0]].ny : l0.blk[r.blk[0]].nx;
  }
  D.vec = vec;
  D.nbm = gm;
  D.m1 = (int)(std::find(mblk.begin(), mblk.end(), 1) - mblk.begin());
  int st;
  if (!f64) {
    // the systems with the smallest -(lambda + sigma): up to LOW_SPAN times the smallest nonzero one, 1/64 of
    // all at most (kern_direct.cu, k_tri_low; rows of longer systems do not fit its CTA). Of all wavenumbers of the
    // problem, so that a plan that holds a range of them solves the same systems the same way
    constexpr double LOW_SPAN = 256.0;
    std::vector<std::pair<double, int>> by;
    std::vector<unsigned char> low((size_t)P->nz * M, 0);
    std::vector<int> smooth(M);  // slots from the smallest -lambda up
    for (int k = 0; k < M; ++k) smooth[k] = k;
    std::stable_sort(smooth.begin(), smooth.end(), [&](int a, int b) { return D.lam[a] > D.lam[b]; });
    const std::vector<double> sigma = all_shifts(P);
    const auto value = [&](int q, int k) { return -(sigma[q] * D.cscale + D.lam[k]); };
    double least = INFINITY;
    for (int q = 0; q < P->nzt; ++q)
      for (int k : smooth)
        if (value(q, k) > 0.0) {
          least = std::min(least, value(q, k));
          break;
        }
    if (N <= 512)
      for (int q = 0; q < P->nzt; ++q)
        for (int k : smooth) {
          if (value(q, k) > LOW_SPAN * least) break;
          by.push_back({value(q, k), q * M + k});
        }
    std::sort(by.begin(), by.end());
    by.resize(std::min(by.size(), (size_t)P->nzt * M / 64));
    std::vector<int> list;
    for (const auto& v : by) {
      const int l = v.second / M - P->q0;
      if (l < 0 || l >= P->nz) continue;
      list.push_back(l * M + v.second % M);
      low[list.back()] = 1;
    }
    D.nlow = (int)list.size();
    if ((st = up_vec(P, &D.d_lam64, D.lam)) || (st = up_vec(P, &D.d_tri64, tri)) ||
        (st = up_vec(P, &D.d_lowlist, list)) || (st = up_vec(P, &D.d_low, low)))
      return st;
  }
  if ((st = up_inner(P, &D.d_tw, tw)) || (st = up_inner(P, &D.d_lam, D.lam)) || (st = up_inner(P, &D.d_tri, tri)) ||
      (st = up_vec(P, &D.d_perm, perm)) || (st = up_vec(P, &D.d_base, base)) || (st = up_vec(P, &D.d_mblk, mblk)) ||
      (st = up_vec(P, &D.d_mstr, mstr)))
    return st;
  return SNAC_OK;
}

// Entries of the transforms as the line kernels scale them (direct_dev.cuh): forward F[kappa][m], inverse
// B[m][kappa], B F = 2 M. From one table of 2 cos(pi t / 4M) or 2 sin(pi t / 4M), t < 8M: the interfaces of the L
// of 512 x 512 cells need 4e5 entries.
struct Entries {
  int kind, M;
  std::vector<double> c, s;
  Entries(int kind_, int M_) : kind(kind_), M(M_) {
    const bool cosine = kind != KIND_DD && kind != KIND_DN, sine = !cosine || kind == KIND_PP;
    for (int t = 0; t < 8 * M; ++t) {
      if (cosine) c.push_back(2.0 * std::cos(M_PI * t / (4.0 * M)));
      if (sine) s.push_back(2.0 * std::sin(M_PI * t / (4.0 * M)));
    }
  }
  double fwd(int kap, int m) const {
    const long long T = 8LL * M;
    switch (kind) {
      case KIND_PP: return kap <= M / 2 ? c[8LL * kap * m % T] : -s[8LL * (M - kap) * m % T];
      case KIND_NN: return c[2 * (2LL * m + 1) * kap % T];
      case KIND_DD: return s[2 * (2LL * m + 1) * (M - kap) % T];
      case KIND_ND: return c[(2LL * m + 1) * (2LL * kap + 1) % T];
      default: return s[(2LL * m + 1) * (2LL * (M - 1 - kap) + 1) % T];
    }
  }
  double bwd(int m, int kap) const {
    const double f = fwd(kap, m);
    const bool half = (kind == KIND_PP && (kap == 0 || kap == M / 2)) || ((kind == KIND_NN || kind == KIND_DD) && kap == 0);
    return half ? 0.5 * f : f;
  }
};

// The matrices between end values, jumps and fluxes.
int build_iface(snac_plan* P, const Layout& L) {
  DirectPlan& D = P->direct;
  IfaceTab& I = D.it;
  I.k = (int)L.cells.size();
  if (I.k == 0) return SNAC_OK;
  std::map<int, int> end_of;  // 2 piece + end -> number
  for (size_t p = 0; p < L.pc.size(); ++p)
    for (int e = 0; e < 2; ++e)
      if (L.pc[p].iface[e]) {
        const int u = I.nends++;
        end_of[(int)(2 * p + e)] = u;
        I.ep[u] = (int)p;
        I.ee[u] = e;
        I.eo[u + 1] = I.eo[u] + D.pc[p].M;
      }
  I.E = I.eo[I.nends];
  for (int l = 0; l < P->nz; ++l)
    if (P->singular && P->sigma[l] == 0.0) I.qs = l;
  for (size_t p = 0; p < L.pc.size(); ++p)
    if (D.pc[p].pin) I.sp[I.ns++] = (int)p;
  I.kk = I.k + I.ns;
  std::vector<double> Y((size_t)I.E * I.kk, 0.0), Z((size_t)I.kk * I.E, 0.0);
  std::vector<Entries> en;
  for (const DirectTab& T : D.pc) en.emplace_back(T.kind, T.cls == LINES_DENSE ? 0 : T.M);
  for (int j = 0; j < I.k; ++j) {
    const IfaceCell& c = L.cells[j];
    I.cells.push_back({{end_of[2 * c.pa + 1], end_of[2 * c.pb]}, {c.ma, c.mb}, {-c.ca, c.cb}});
    for (int side = 0; side < 2; ++side) {
      const int p = side == 0 ? c.pa : c.pb, m = side == 0 ? c.ma : c.mb;
      const int u = end_of[2 * p + (side == 0 ? 1 : 0)];
      const DirectTab& T = D.pc[p];
      for (int k = 0; k < T.M; ++k) {
        Y[(size_t)(I.eo[u] + k) * I.kk + j] = (side == 0 ? -1.0 : 1.0) * (T.cls == LINES_DENSE ? T.B[(size_t)m * T.M + k] : en[p].bwd(m, k));
        Z[(size_t)j * I.E + I.eo[u] + k] = (side == 0 ? -c.ca : c.cb) * (T.cls == LINES_DENSE ? T.F[(size_t)k * T.M + m] : en[p].fwd(k, m));
      }
    }
  }
  const size_t w = P->precision == SNAC_FP64 ? sizeof(double) : sizeof(float);
  int st;
  if ((st = up_vec(P, &I.d_Y, Y)) || (st = up_inner(P, &I.d_Z, Z)) ||
      (st = plan_alloc(P, &I.d_ends, (size_t)P->nz * I.E * w)) || (st = plan_alloc(P, &I.d_alpha, (size_t)P->nz * IFACE_MAX_ENDS * w)) ||
      (st = plan_alloc(P, &I.d_num, (size_t)P->nz * IFACE_MAX_ENDS * w)))
    return st;
  I.Zh.swap(Z);
  return SNAC_OK;
}

// The interface systems are dense: k^2 values per wavenumber kept, k^2 (E + k) operations to set them up.
bool iface_affordable(const snac_plan* P, const Layout& L) {
  const double k = (double)L.cells.size();
  double E = 0.0;
  int ends = 0;
  for (const Piece& p : L.pc)
    for (int e = 0; e < 2; ++e)
      if (p.iface[e]) {
        int m = 0;
        for (int b : p.rows[0].blk) m += L.axis == 0 ? P->lev[0].blk[b].nx : P->lev[0].blk[b].ny;
        E += m;
        ++ends;
      }
  return ends <= IFACE_MAX_ENDS && (int)L.pc.size() <= IFACE_MAX_ENDS && k <= 1024 && E <= 8192 &&
         P->nz * k * k <= 64e6 && P->nz * k * k * (E + k) <= 4e10;
}

}  // namespace

// Of the two plane axes the cheaper one is transformed, x where they tie (its lines are contiguous).
static int build_direct(snac_plan* P, const std::vector<FaceKinds>& faces) {
  Layout best;
  double least = INFINITY;
  for (int t = 0; t < 2; ++t) {
    Layout L;
    if (!pieces_along(P, faces, t, L) || !iface_affordable(P, L)) continue;
    const double cost = layout_cost(P, L);
    if (cost < 0.0 || cost >= least) continue;
    best = L;
    least = cost;
  }
  if (!std::isfinite(least)) return SNAC_OK;
  DirectPlan& D = P->direct;
  int soff = 0, st;
  for (const Piece& p : best.pc) {
    D.pc.emplace_back();
    if ((st = build_piece(P, p, best.axis, soff, D.pc.back()))) return st;
    soff += D.pc.back().M * D.pc.back().N;
  }
  if ((st = build_iface(P, best))) return st;
  for (DirectTab& d : D.pc) {
    std::vector<double>().swap(d.F);
    std::vector<double>().swap(d.B);
  }
  D.on = true;
  return SNAC_OK;
}

static int finish_direct(snac_plan* P) {
  DirectPlan& D = P->direct;
  const bool f64 = P->precision == SNAC_FP64;
  const size_t w = f64 ? sizeof(double) : sizeof(float);
  int st;
  std::vector<int> qrow(P->nz), qof;
  int* d_qof = nullptr;
  std::map<int, int> seen;  // wavenumbers q and n - q of the real DFT have one eigenvalue
  for (int l = 0; l < P->nz; ++l) {
    const int q = P->q0 + l;
    const auto it = seen.emplace(P->kind == KIND_PP ? std::min(q, P->nzt - q) : q, (int)qof.size());
    if (it.second) qof.push_back(l);
    qrow[l] = it.first->second;
  }
  if ((st = up_vec(P, &D.d_qrow, qrow)) || (st = up_vec(P, &d_qof, qof))) return st;
  if (D.it.k && (st = plan_alloc(P, (void**)&D.it.d_KT, qof.size() * D.it.kk * (size_t)D.it.kk * sizeof(double)))) return st;
  if (!P->onchip) {
    for (DirectTab& T : D.pc)
      if ((st = plan_alloc(P, &T.d_fac, qof.size() * (size_t)T.M * T.N * w))) return st;
  } else {
    // the cells' places in the on-chip buffer, and the pieces' arguments
    std::vector<unsigned> off(P->lev[0].ncell, 0u);
    const auto place = [&](auto tag) {
      using T = decltype(tag);
      std::vector<DirectArgs<T>> args;
      size_t base = 0;
      for (const DirectTab& d : D.pc) {
        const DirectArgs<T> A = direct_args<T>(P, d);
        args.push_back(A);
        const PlaneShape S = plane_shape(A.F, A.M, A.N, A.cls);
        auto row = [&](int p) { return (size_t)(p / A.F.l1) * S.s1 + (size_t)(p % A.F.l1) * S.rp; };
        const bool flip = d.kind == KIND_DD || d.kind == KIND_DN;
        for (int n = 0; n < d.N; ++n)
          for (int m = 0; m < d.M; ++m) {
            const long long c = d.base[(size_t)n * d.nbm + d.mblk[m]] + (long long)m * d.mstr[n];
            size_t o;
            if (d.cls == LINES_PAIR) {
              const int t = d.kind == KIND_PP ? m : ((m & 1) ? d.M - 1 - (m >> 1) : m >> 1);
              o = 2 * (row(t) + (n >> 1)) + (n & 1);
            } else {
              o = 2 * (row((m & 1) ? (d.M - 1 - m) >> 1 : m >> 1) + n) + (m & 1);
            }
            off[c] = (unsigned)(base + o) | (flip && (m & 1) ? 0x80000000u : 0u);
          }
        base += S.buf;
      }
      return plan_upload(P, &D.d_args, args.data(), args.size() * sizeof(DirectArgs<T>));
    };
    if ((st = f64 ? place(double{}) : place(float{})) || (st = up_vec(P, &D.d_celloff, off))) return st;
  }
  // on the private stream, like every other device work of plan creation
  const cudaStream_t cs = P->setup_stream;
  cudaError_t e = cudaSuccess;
  for (DirectTab& T : D.pc) {
    if (e == cudaSuccess && T.d_fac) e = launch_tri_factor(P, T, d_qof, (int)qof.size(), cs);
    for (std::vector<int>* v : {&T.base, &T.mblk, &T.mstr}) std::vector<int>().swap(*v);
  }
  if (e == cudaSuccess && D.it.k) e = setup_iface(P, d_qof, (int)qof.size(), D.it.qs < 0 ? -1 : qrow[D.it.qs], cs);
  if (e == cudaSuccess) e = cudaStreamSynchronize(cs);
  if (e != cudaSuccess) {
    cudaGetLastError();
    set_error(std::string("setting up the direct solves failed: ") + cudaGetErrorString(e));
    return e == cudaErrorMemoryAllocation ? SNAC_ERR_OOM : SNAC_ERR_CUDA;
  }
  return SNAC_OK;
}

size_t direct_interface_bytes(const snac_plan* P, const std::vector<FaceKinds>& faces) {
  const size_t w = P->precision == SNAC_FP64 ? sizeof(double) : sizeof(float);
  size_t most = 0;
  for (int t = 0; t < 2; ++t) {
    Layout L;
    if (!pieces_along(P, faces, t, L) || L.cells.empty() || !iface_affordable(P, L)) continue;
    size_t E = 0, M = 0;
    for (const Piece& p : L.pc) {
      const size_t m = piece_widths(P, p, t, true).size();
      M += m;
      for (int e = 0; e < 2; ++e) E += p.iface[e] ? m : 0;
    }
    const size_t kk = L.cells.size() + L.pc.size(), nz = (size_t)P->nz, rows = P->kind == KIND_PP ? nz / 2 + 1 : nz;
    // kept: inverses, Y, Z, end values, pinned unknowns; while they are set up: responses and their cosine sums, a
    // second Z, the cells
    most = std::max(most, rows * kk * kk * sizeof(double) + E * kk * (sizeof(double) + w) + nz * E * w +
                              2 * nz * IFACE_MAX_ENDS * w + rows * (M + L.pc.size()) * sizeof(double4) +
                              E * kk * sizeof(double) + rows * 4 * E * sizeof(double) + kk * sizeof(IfaceCellDev));
  }
  return most;
}

int setup_direct(snac_plan* P, const std::vector<FaceKinds>& faces) {
  if (P->lev[0].ncell >= (1LL << 31)) return SNAC_OK;
  const size_t mark = P->allocs.size(), bytes = P->bytes;
  int st;
  try {
    st = build_direct(P, faces);
    if (st == SNAC_OK && P->direct.on && P->onchip && direct_onchip_smem(P) > (size_t)BOTTOM_MAX_SMEM) st = NOT_DIRECT;
    if (st == SNAC_OK && P->direct.on) st = finish_direct(P);
  } catch (const std::bad_alloc&) {
    st = SNAC_ERR_OOM;
  }
  if (st != NOT_DIRECT && st != SNAC_ERR_OOM) return st;
  set_error("");
  for (size_t k = mark; k < P->allocs.size(); ++k) cudaFree(P->allocs[k]);
  P->allocs.resize(mark);
  P->bytes = bytes;
  P->direct = DirectPlan{};
  return SNAC_OK;
}

size_t direct_onchip_smem(const snac_plan* P) {
  const DirectPlan& D = P->direct;
  size_t el = 0;
  for (const DirectTab& d : D.pc) el += plane_shape(d.fft, d.M, d.N, d.cls).buf;
  return onchip_elements(el, BOTTOM_THREADS) * (P->precision == SNAC_FP64 ? sizeof(double) : sizeof(float)) +
         iface_doubles(D.it.E, D.it.kk, BOTTOM_THREADS) * sizeof(double);
}

}  // namespace snac
