"""Direct solves of the reduced equations (a transform along a uniform plane axis and tridiagonal systems
along the other, on an assembled rectangle or on several that meet along parts of their sides), through
the C ABI.

``mode_solve`` of a random right-hand side is checked wavenumber by wavenumber with the oracle's plane
operator. The bound: the transforms and the elimination are backward stable, so the solution carries
errors of a few units of rounding u times the largest value of the plane (the transforms mix the cells
of a line) and the residual those times the row sums of |A|, plus a few u of the right-hand side. Each
of the two transforms adds about log2(M) roundings; 16 u per level covers them and the approximate
reciprocals of the elimination (4e-15 relative in FP64, 2 units in the last place in FP32)."""
import numpy as np
import pytest

from oracle import grid as ogrid
from oracle import solve as osv
from oracle import transforms as T
from paper_2106_03583_gb300 import inputs

from gpu_util import dev, host, plan, rel
from layouts import Z_PAIRS, homogeneous_along

pytestmark = pytest.mark.gpu


def rects(layout, nx, ny):
    hx, hy, tx, ty = nx // 2, ny // 2, nx // 3, ny // 3
    return {# T junction, U, Z, and a ring around a hole (a square cylinder): several rectangles
            "T": [(0, tx, 0, hy), (tx, 2 * tx, 0, hy), (2 * tx, nx, 0, hy), (tx, 2 * tx, hy, ny)],
            "U": [(0, tx, 0, hy), (tx, 2 * tx, 0, hy), (2 * tx, nx, 0, hy), (0, tx, hy, ny), (2 * tx, nx, hy, ny)],
            "Z": [(0, tx, 0, hy), (tx, 2 * tx, 0, hy), (tx, 2 * tx, hy, ny), (2 * tx, nx, hy, ny)],
            "O": [(i * tx, (i + 1) * tx, j * ty, (j + 1) * ty) for j in range(3) for i in range(3) if (i, j) != (1, 1)],
            "1": [(0, nx, 0, ny)], "1x2": [(0, hx, 0, ny), (hx, nx, 0, ny)], "2x1": [(0, nx, 0, hy), (0, nx, hy, ny)],
            "L": [(0, hx, 0, hy), (hx, nx, 0, hy), (0, hx, hy, ny)],
            # blocks listed out of order
            "2x2": [(hx, nx, 0, hy), (0, hx, hy, ny), (0, hx, 0, hy), (hx, nx, hy, ny)]}[layout]


def build(layout, nx, ny, xfac, yfac, walls, zpair="NN", nz=6, per=(False, False)):
    wb = dict(zip(("x-", "x+", "y-", "y+"), walls))
    return inputs.make_blocks(inputs.tanh_faces(nx, 0, xfac, 0.0, 1.3), inputs.tanh_faces(ny, 0, yfac, 0.0, 1.0),
                              np.linspace(0.0, 0.8, nz + 1), rects(layout, nx, ny), wb, Z_PAIRS[zpair], periodic=per)


# layout, nx, ny, stretching of x and y, walls, z pair, periodic axes
DIRECT = [
    ("1", 64, 40, 0.0, 1.5, "DDNN", "PP", (False, False)),      # x lines, DST-II; one CTA per wavenumber
    ("2x2", 48, 48, 0.0, 1.5, "NNNN", "NN", (False, False)),    # singular, four blocks
    ("1x2", 80, 16, 0.0, 1.0, "NDDD", "DD", (False, False)),    # DCT-IV, factor 5
    ("2x1", 28, 36, 0.0, 1.2, "DNNN", "ND", (False, False)),    # DST-IV, factor 7
    ("1", 40, 64, 1.3, 0.0, "DNND", "DN", (False, False)),      # y lines, DCT-IV
    ("2x2", 40, 48, 1.3, 0.0, "DDNN", "PP", (False, False)),    # y lines, DCT-II
    ("1x2", 48, 40, 0.0, 1.2, "DDDN", "NN", (True, False)),     # periodic x across two blocks
    ("1", 24, 32, 1.1, 0.0, "DNNN", "DD", (False, True)),       # periodic y of one block, x tridiagonal
    ("1", 160, 128, 0.0, 1.0, "NNDD", "PP", (False, False)),    # planes of three passes, DCT-II
    ("2x2", 160, 160, 0.0, 1.0, "DNNN", "NN", (False, False)),  # DST-IV
    ("1x2", 128, 144, 1.1, 0.0, "DDDD", "DD", (False, False)),  # y lines, factor 9
    ("2x2", 144, 96, 1.1, 0.0, "NNND", "PP", (False, False)),   # y lines, DCT-IV
    ("1", 4, 45, 0.0, 1.0, "DDNN", "PP", (False, False)),       # the shortest lines, odd number of them
    ("1", 45, 4, 1.0, 0.0, "NNDD", "NN", (False, False)),       # the same along y
    ("1", 14, 18, 0.0, 0.8, "NNNN", "PP", (False, False)),      # singular, one multigrid level
    ("2x1", 32, 576, 0.0, 1.0, "DNDN", "PP", (True, False)),    # more than 512 rows
    ("1", 32, 1088, 0.0, 1.0, "DDNN", "NN", (False, False)),    # more than 1024 rows
    ("1", 1024, 16, 0.0, 1.0, "NNNN", "DD", (False, False)),    # long lines
    # several pieces; one CTA per wavenumber
    ("L", 32, 32, 0.0, 0.0, "DDNN", "NN", (False, False)),
    ("L", 48, 40, 0.0, 1.2, "NNNN", "PP", (False, False)),      # singular
    ("T", 48, 32, 0.0, 1.0, "NNDN", "NN", (False, False)),      # one singular piece in a regular problem
    ("U", 72, 24, 0.0, 0.7, "DNNN", "ND", (False, False)),      # two interfaces on one side
    ("Z", 48, 28, 0.0, 0.7, "NNNN", "NN", (False, False)),      # singular pieces
    ("O", 48, 48, 0.0, 0.0, "NNNN", "PP", (False, False)),      # a hole, four pieces, singular
    ("L", 40, 64, 1.1, 0.0, "NDND", "DD", (False, False)),      # y lines
    ("T", 48, 32, 0.0, 1.0, "DDNN", "PP", (True, False)),       # one piece periodic along its lines
    # several pieces; planes of several passes
    ("L", 256, 160, 0.0, 1.0, "DNNN", "NN", (False, False)),
    ("L", 160, 256, 0.0, 0.0, "NNNN", "PP", (False, False)),
    ("O", 192, 192, 0.0, 0.0, "DNNN", "ND", (False, False)),
    ("T", 192, 320, 1.0, 0.0, "NNNN", "NN", (False, False)),    # y lines, singular
    # dense transforms: axes clustered both ways, or a length with a prime factor 11
    ("1", 160, 96, 1.3, 1.5, "DNNN", "DN", (False, False)),
    ("2x2", 96, 160, 1.0, 1.0, "NNNN", "NN", (False, False)),   # singular, x lines
    ("1", 88, 96, 0.0, 1.2, "NNDN", "DD", (False, False)),
    ("L", 160, 128, 1.0, 1.0, "DDNN", "NN", (False, False)),
    ("T", 240, 128, 1.0, 1.0, "NNNN", "PP", (False, False)),    # singular
    # segments of 16 rows, 32 / 16 / 8 systems per CTA: a last CTA not full, a last segment not full, 17 segments,
    # the most segments, and the end values of 17 segments (singular)
    ("1", 72, 128, 0.0, 1.0, "NNNN", "NN", (False, False)),
    ("1", 128, 72, 0.0, 1.0, "DDNN", "PP", (False, False)),
    ("1", 40, 264, 0.0, 1.0, "NNDN", "DD", (False, False)),
    ("1", 16, 1024, 0.0, 1.0, "DNNN", "NN", (False, False)),
    ("L", 64, 544, 0.0, 1.0, "NNNN", "NN", (False, False)),
]


def _passes(pl):
    st = pl.kernel_stats()
    return st["lines_forward"]["launches"] + st["onchip"]["launches"], st


def _check_modes(blocks, precision, shift=0.0, modes=None, dense=False):
    import torch
    g = ogrid.Grid(blocks, shift=shift)
    pl = plan(blocks, precision=precision, shift=shift, modes=modes)
    q0, q1 = pl.mode_range
    rng = np.random.default_rng(5)
    F = rng.standard_normal((q1 - q0, g.plane.n)).astype(np.float32 if precision == "mixed" else np.float64)
    F = F.astype(np.float64)
    lam = T.eigenvalues(g.kind, g.nz)[q0:q1] / g.dz ** 2 + shift
    sing = [g.singular and lam[k] == 0.0 for k in range(q1 - q0)]
    for k in range(q1 - q0):
        if sing[k]:
            F[k] -= np.dot(g.plane.area, F[k]) / g.plane.area.sum()
    u = torch.empty(F.size, dtype=pl.inner_dtype, device="cuda")
    info = pl.mode_solve(dev(F.ravel(), pl.inner_dtype), u, target=0.0)
    n, st = _passes(pl)
    U = host(u).reshape(F.shape)
    eps = 2.0 ** -24 if precision == "mixed" else 2.0 ** -53
    absrow = np.asarray(abs(g.plane.A).sum(axis=1)).ravel()
    nmax = max(len(np.unique(g.plane.gx)), len(np.unique(g.plane.gy)))
    # (several pieces: the dense interface systems add sums of up to nmax terms, 1/2 u sqrt(nmax) each way, and the
    # solution is formed twice)
    pieces = len(np.unique(g.plane.gx)) * len(np.unique(g.plane.gy)) != g.plane.n
    pieces = pieces or dense   # (the same for dense transforms: sums of nmax terms twice)
    c = 16 * eps * (np.log2(nmax) + 4) * (1 + (2 + 0.25 * np.sqrt(nmax)) * pieces)
    for k in range(q1 - q0):
        r = F[k] - (g.plane.A @ U[k] + lam[k] * U[k])
        bound = c * (np.linalg.norm(absrow + abs(lam[k])) * np.abs(U[k]).max() + np.linalg.norm(F[k]))
        assert np.linalg.norm(r) <= bound, (k, np.linalg.norm(r) / bound)
    assert n >= 1 and st["smooth"]["launches"] == st["fused_up"]["launches"] == st["bottom"]["launches"] == 0
    assert info["total_cycles"] == q1 - q0 and np.all(pl.mode_cycles() == 1)
    pl.close()


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("case", DIRECT, ids=lambda c: "-".join(map(str, c[:6])))
def test_direct_mode_solve(case, precision):
    layout, nx, ny, xf, yf, walls, zp, per = case
    _check_modes(build(layout, nx, ny, xf, yf, walls, zp, per=per), precision, dense=(xf > 0 and yf > 0) or nx % 11 == 0)


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_direct_mode_solve_shift_and_range(precision):
    _check_modes(build("2x2", 48, 40, 0.0, 1.5, "NNNN", "NN"), precision, shift=-3.0)
    _check_modes(build("1", 160, 128, 0.0, 1.0, "NNNN", "NN", nz=10), precision, modes=(3, 8))
    _check_modes(build("2x2", 48, 40, 0.0, 1.5, "NNNN", "NN", nz=10), precision, modes=(0, 5))


@pytest.mark.parametrize("kw,case", [
    ({}, ("L", 32, 32, 1.0, 1.0, "DDNN")), ({}, ("1", 32, 32, 1.0, 1.0, "DDNN")),
    ({}, ("1", 44, 32, 0.0, 1.0, "DDNN")),                       # 11 divides the uniform axis
    ({"onchip": False}, ("1", 32, 32, 0.0, 0.0, "DDNN")), ({"nu1": 1}, ("1", 32, 32, 0.0, 0.0, "DDNN")),
    ({"bottom_cells": 512}, ("1", 32, 32, 0.0, 0.0, "DDNN")), ({"max_coarse": 16}, ("1", 32, 32, 0.0, 0.0, "DDNN"))])
def test_multigrid_keeps_the_other_plans(kw, case):
    """Layouts that are not separable, and plans with a schedule of their own, run V-cycles."""
    import torch
    blocks = build(*case)
    g = ogrid.Grid(blocks)
    pl = plan(blocks, **kw)
    F = np.random.default_rng(6).standard_normal((g.nz, g.plane.n))
    u = torch.empty(F.size, dtype=torch.float64, device="cuda")
    info = pl.mode_solve(dev(F.ravel()), u, target=1e-8)
    assert info["total_cycles"] > 2 * g.nz and pl.kernel_stats()["lines_forward"]["launches"] == 0
    pl.close()


@pytest.mark.parametrize("homog", [2, 0, 1])
@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("case", [DIRECT[1], DIRECT[7], DIRECT[9], DIRECT[10], DIRECT[19], DIRECT[23], DIRECT[26]], ids=lambda c: "-".join(map(str, c[:6])))
def test_direct_solve_vs_oracle(case, precision, homog):
    """Whole solves of separable layouts, the homogeneous direction along each caller axis."""
    import torch
    layout, nx, ny, xf, yf, walls, zp, per = case
    blocks = build(layout, nx, ny, xf, yf, walls, zp, per=per)
    f = inputs.divergence_rhs(blocks, 8)
    ref, _ = osv.solve(blocks, f)
    rb, rf, back = homogeneous_along(blocks, f, homog)
    pl = plan(rb, precision=precision, homog_axis=homog)
    p = torch.zeros(len(f), dtype=torch.float64, device="cuda")
    info = pl.solve(dev(rf), p, tol=1e-10)
    assert info["status"] == 0 and info["total_cycles"] == info["outer_iters"] * g_nz(blocks)
    assert osv.rel_residual(blocks, f, back(host(p))) <= 1.01e-10
    assert rel(back(host(p)), ref) <= 1e-9
    pl.close()


def g_nz(blocks):
    return blocks[0]["hi"][2] - blocks[0]["lo"][2] + 1


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("case", [DIRECT[0], DIRECT[8]], ids=lambda c: "-".join(map(str, c[:6])))
def test_direct_mode_solve_reports_nonfinite_input(case, precision):
    import torch
    from paper_2106_03583_gb300 import snac
    layout, nx, ny, xf, yf, walls, zp, per = case
    blocks = build(layout, nx, ny, xf, yf, walls, zp, per=per)
    pl = plan(blocks, precision=precision)
    n = pl.nmodes * pl.ncell
    f = torch.ones(n, dtype=pl.inner_dtype, device="cuda")
    u = torch.empty_like(f)
    for bad in (float("nan"), float("inf")):
        f[n // 2] = bad
        with pytest.raises(snac.SnacError) as e:
            pl.mode_solve(f, u, target=1e-3)
        assert e.value.name == "NONFINITE"
    f[n // 2] = 1.0
    assert pl.mode_solve(f, u, target=1e-3)["status"] == 0
    pl.close()


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("case", [("T", 48, 32, 0.0, 1.0, "NNDN", "NN"), ("L", 32, 32, 0.0, 1.0, "NNDN", "PP"),
                                  ("T", 192, 320, 0.0, 1.0, "NNDN", "NN"), ("L", 64, 544, 0.0, 1.0, "NNDN", "NN")],
                         ids=lambda c: "-".join(map(str, c[:6])))
def test_direct_solve_with_a_nearly_singular_piece(case, precision):
    """A small Helmholtz shift leaves a piece without Dirichlet faces nearly singular while the whole problem is
    not: as many steps as without a shift, and the solution of a sparse factorisation of the oracle's planes (the
    oracle's own V-cycles stop at a residual of 0.4 on the 64 x 544 plane)."""
    import torch
    from scipy.sparse import identity
    from scipy.sparse.linalg import spsolve
    blocks = build(*case)
    f = inputs.divergence_rhs(blocks, 8)
    steps = []
    for shift in (0.0, -1e-13, -1e-8, -1e-4, -1e-2, -1.0, -10.0):
        pl = plan(blocks, precision=precision, shift=shift)
        p = torch.zeros(len(f), dtype=torch.float64, device="cuda")
        info = pl.solve(dev(f), p, tol=1e-10)
        pl.close()
        assert info["status"] == 0
        steps.append(info["outer_iters"])
        assert osv.rel_residual(blocks, f, host(p), shift=shift) <= 1.01e-10
        if shift == -1e-8:
            g = ogrid.Grid(blocks, shift)
            sigma = T.eigenvalues(g.kind, g.nz) / g.dz ** 2 + shift
            F = T.forward(g.kind, g.to_planes(f))
            P = [spsolve((g.plane.A + s * identity(g.plane.n)).tocsc(), x) for s, x in zip(sigma, F)]
            assert rel(host(p), g.from_planes(T.backward(g.kind, np.array(P)))) <= 1e-9
    assert max(steps) <= steps[0] + 1


@pytest.mark.parametrize("unit", [2.0 ** -250, 2.0 ** 266])
def test_dense_transforms_in_any_unit_of_length(unit):
    """Cell widths times a power of two: the same solution times its square, to rounding."""
    import torch
    out = []
    for scale in (1.0, unit):
        blocks = build("1", 160, 96, 1.3, 1.5, "DNNN", "DN")
        f = inputs.divergence_rhs(blocks, 8)
        for b in blocks:
            b["dx"] = tuple(np.asarray(w) * scale for w in b["dx"])
        pl = plan(blocks)
        p = torch.zeros(len(f), dtype=torch.float64, device="cuda")
        assert pl.solve(dev(f), p, tol=1e-10)["outer_iters"] == 1 and pl.kernel_stats()["lines_forward"]["launches"] == 1
        pl.close()
        out.append(host(p))
    assert rel(out[1] / unit ** 2, out[0]) <= 1e-13


@pytest.mark.parametrize("case", [DIRECT[0], DIRECT[8], DIRECT[26]], ids=lambda c: "-".join(map(str, c[:6])))
def test_loose_tolerance_takes_one_residual_pass(case):
    """A mixed solve that one direct step finishes: the residual before it is f, the one after it FP64, and no
    float-float pass between."""
    import torch
    layout, nx, ny, xf, yf, walls, zp, per = case
    blocks = build(layout, nx, ny, xf, yf, walls, zp, per=per)
    f = inputs.divergence_rhs(blocks, 8)
    pl = plan(blocks, precision="mixed")
    p = torch.zeros(len(f), dtype=torch.float64, device="cuda")
    info = pl.solve(dev(f), p, tol=1e-3)
    st = pl.kernel_stats()
    assert info["status"] == 0 and info["outer_iters"] == 1
    assert st["field3d_ff"]["launches"] == 0 and st["field3d"]["launches"] == 2   # the statistics of f, the residual
    assert osv.rel_residual(blocks, f, host(p)) <= 1.01e-3
    pl.close()


@pytest.mark.parametrize("case", [("1", 32, 768, 0.0, 2.0, "DDNN", "PP"), ("1", 64, 1024, 0.0, 2.0, "DDNN", "PP"),
                                  ("L", 64, 544, 0.0, 1.0, "NNDN", "NN")], ids=lambda c: "-".join(map(str, c[:6])))
def test_mixed_step_near_the_tolerance_starts_from_the_fp64_residual(case):
    """A step from a residual within twice the tolerance 1e-10 reduces it by 6e-7 or more, to 1.2e-16, if it is the
    FP64 residual: what is left is the FP64 rounding of the residual of these clustered axes, below 2e-12. From a
    float-float residual it would be about 1e-11."""
    import torch
    layout, nx, ny, xf, yf, walls, zp = case
    blocks = build(layout, nx, ny, xf, yf, walls, zp, nz=8)
    f = inputs.divergence_rhs(blocks, 1)
    pl = plan(blocks, precision="mixed")
    p = torch.zeros(len(f), dtype=torch.float64, device="cuda")
    info = pl.solve(dev(f), p, tol=1e-10)
    assert info["status"] == 0 and info["outer_iters"] == 3 and info["rel_res"] <= 2e-12
    pl.close()


@pytest.mark.parametrize("case", [DIRECT[8], DIRECT[26], DIRECT[0]], ids=lambda c: "-".join(map(str, c[:6])))
def test_mixed_range_plan_solves_as_the_whole_plan(case):
    """A plan that holds some wavenumbers takes the smoothest systems of the whole problem in FP64, as the whole plan
    does: the same solutions bit for bit."""
    import torch
    layout, nx, ny, xf, yf, walls, zp, per = case
    blocks = build(layout, nx, ny, xf, yf, walls, zp, nz=12, per=per)
    whole, n = plan(blocks, precision="mixed"), 12
    F = torch.from_numpy(np.random.default_rng(7).standard_normal((n, whole.ncell)).astype(np.float32)).cuda()
    u = torch.empty_like(F)
    whole.mode_solve(F, u, target=0.0)
    for a, b in ((0, 5), (5, 12)):
        part = plan(blocks, precision="mixed", modes=(a, b))
        v = torch.empty((b - a, whole.ncell), dtype=torch.float32, device="cuda")
        part.mode_solve(F[a:b].contiguous(), v, target=0.0)
        assert torch.equal(v, u[a:b])
        part.close()
    whole.close()


# two rows of blocks around a periodic axis whose rings are met at different blocks; interfaces of 1024 cells with two
# pinned pieces (1026 unknowns: more than the threads of the interface kernel)
@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("case", [("2x2", 48, 40, 0.0, 1.2, "NNDN", "NN", 6, (True, False)),
                                  ("2x2", 160, 128, 0.0, 1.0, "NNNN", "PP", 6, (True, False)),
                                  ("2x2", 40, 48, 1.1, 0.0, "DNNN", "DD", 6, (False, True)),
                                  ("L", 2048, 2048, 0.0, 0.0, "NNNN", "NN", 4, (False, False))],
                         ids=lambda c: "-".join(map(str, c[:6])))
def test_direct_mode_solve_rings_and_long_interfaces(case, precision):
    layout, nx, ny, xf, yf, walls, zp, nz, per = case
    _check_modes(build(layout, nx, ny, xf, yf, walls, zp, nz=nz, per=per), precision)
