"""Plan creation on the host (no GPU: tests/fake_cudart.cpp stands in for the CUDA runtime)."""
import pytest

import fake_cuda

# an L of three blocks, a rectangle clustered both ways (dense transforms), small planes of one piece and of
# three, and a plan that keeps its V-cycles (a prime axis)
LAYOUTS = """
def face(n, f):
    return inputs.tanh_faces(n, 0, f, 0.0, 1.0)
def problem(rects, nx, ny, nz=8, xf=0.0, yf=0.0, z=("N", "N"), walls="DNNN"):
    return inputs.make_blocks(face(nx, xf), face(ny, yf), np.linspace(0.0, 1.0, nz + 1), rects,
                              dict(zip(("x-", "x+", "y-", "y+"), walls)), z)
L = lambda n: [(0, n, 0, n), (n, 2 * n, 0, n), (0, n, n, 2 * n)]
PROBLEMS = {
    "L": lambda: problem(L(80), 160, 160, z=("P", "P")), "L on chip": lambda: problem(L(16), 32, 32),
    "dense": lambda: problem([(0, 160, 0, 128)], 160, 128, xf=1.0, yf=1.0),
    "on chip": lambda: problem([(0, 32, 0, 32)], 32, 32, yf=1.0),
    "planes": lambda: problem([(0, 160, 0, 128)], 160, 128, yf=1.0),
    "V-cycles": lambda: problem([(0, 416, 0, 416)], 416, 416, xf=1.0, yf=1.0),
}
"""


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_setup_kernels_run_after_the_tables_have_arrived(precision):
    out = fake_cuda.run(LAYOUTS + f"""
out = dict()
for name, make in PROBLEMS.items():
    fake.fake_reset()
    st, h = create(make(), {precision!r})
    out[name] = [st, len(launches()), fake.fake_unordered().decode().split()]
    lib.snac_plan_destroy(h)
""")
    assert sum(n for _, n, _ in out.values()) > 0
    for name, (st, _, unordered) in out.items():
        assert st == 0 and unordered == [], name
    assert len(out) == 6


def test_pencil_kernels_run_after_their_tables_have_arrived():
    out = fake_cuda.run(LAYOUTS + """
st, h = create(PROBLEMS["on chip"]())
buf = (ctypes.c_double * (8 * 1024))()
s = ctypes.c_void_p(8)
halo, n = (ctypes.c_int64 * 4096)(), ctypes.c_int64()
sums = (ctypes.c_double * 5)()
fake.fake_reset()
r = [lib.snac_pencil_setup(h, 0, 1024, halo, 4096, ctypes.byref(n)),
     lib.snac_pencil_residual(h, buf, buf, buf, 0.0, sums, s), lib.snac_pencil_forward(h, 1024, buf, buf, s)]
out = [st, r, len(launches()), fake.fake_unordered().decode().split()]
""")
    assert out[:2] == [0, [0, 0, 0]] and out[2] >= 3 and out[3] == []


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_cell_widths_of_any_size(precision):
    """Widths whose squares or products leave the range of a double: no plan is refused for its eigenvectors, and
    only couplings that are not numbers lose the direct solve."""
    out = fake_cuda.run(LAYOUTS + f"""
out = []
for scale, first, walls in ((1.0, 1.0, "DNDN"), (1e-75, 1.0, "DNDN"), (1e-100, 1.0, "DNDN"), (1e80, 1.0, "DNDN"),
                            (1.0, 1e-160, "DNNN"), (1.0, 1e-160, "NNDN")):
    b = problem([(0, 160, 0, 128)], 160, 128, xf=1.0, yf=1.0, walls=walls)
    for q in b:
        q["dx"] = tuple(np.asarray(w) * scale for w in q["dx"])
        for w in q["dx"][:2]:
            w[0] *= first
    fake.fake_reset()
    st, h = create(b, {precision!r})
    out.append([st, any("k_tri_factor" in n for n in launches())])
    lib.snac_plan_destroy(h)
""")
    assert out == [[0, True]] * 4 + [[0, False]] * 2


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("name", ["L", "L on chip", "dense", "planes"])
def test_direct_setup_out_of_memory(name, precision):
    """A plan whose multigrid fits is created whether the direct solve's tables fit or not, and keeps none of them
    where they do not; every allocation fails once."""
    out = fake_cuda.run(LAYOUTS + f"""
out = []
b = PROBLEMS[{name!r}]()
st, h = create(b, {precision!r})
want = workspace(h)
lib.snac_plan_destroy(h)
n = 0
while True:
    fake.fake_reset()
    before = fake.fake_used()
    fake.fake_fail_after(n)
    st, h = create(b, {precision!r})
    fake.fake_fail_after(-1)
    out.append([st, workspace(h) == fake.fake_used() - before if st == 0 else True, workspace(h) if st == 0 else 0])
    lib.snac_plan_destroy(h)
    out[-1].append(fake.fake_used() == before)
    if out[-1][2] == want:
        break
    n += 1
""")
    status = [o[0] for o in out]
    first = status.index(0)
    assert all(s == -3 for s in status[:first]) and all(s == 0 for s in status[first:])
    assert all(o[1] and o[3] for o in out)
    fallback = out[first:-1]   # plans that kept their V-cycles: the same memory, less than with the tables
    assert len(fallback) >= 8 and len({o[2] for o in fallback}) == 1 and fallback[0][2] < out[-1][2]


def test_setup_reads_nothing_back():
    """The cells' places come from the tables that were uploaded, not from unchecked copies of them."""
    out = fake_cuda.run(LAYOUTS + """
for make in PROBLEMS.values():
    st, h = create(make())
    lib.snac_plan_destroy(h)
out = fake.fake_log().decode().count("read back")
""")
    assert out == 0


@pytest.mark.parametrize("name", ["L", "L on chip", "dense"])
def test_setup_waits_for_no_other_stream(name):
    """cudaFree waits for the whole device: plan creation does without, in stream order."""
    out = fake_cuda.run(LAYOUTS + f"""
st, h = create(PROBLEMS[{name!r}]())
out = [st, fake.fake_log().decode().split().count("cudaFree"), fake.fake_used() == workspace(h)]
""")
    assert out == [0, 0, True]


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("name", ["thin", "L", "T", "dense", "on chip"])
def test_engine_reserves_what_a_plan_takes(name, precision):
    """What an engine has reserved covers the device's memory at its highest, the set-up of the interface systems
    of two long thin rectangles included; where the budget has no room for those, the plan keeps its V-cycles."""
    out = fake_cuda.run(LAYOUTS + f"""
def thin():   # (the Dirichlet face beside an interface rules out rectangles that meet along their short sides)
    b = problem([(0, 84, 0, 4), (0, 84, 4, 8), (84, 168, 4, 8)], 168, 8, nz=4096)
    b[0]["bc"] = (("D", "D"),) + tuple(b[0]["bc"][1:])
    return b
PROBLEMS["thin"] = thin
PROBLEMS["T"] = lambda: problem([(0, 80, 0, 80), (80, 160, 0, 80), (160, 240, 0, 80), (80, 160, 80, 160)], 240, 160, nz=32,
                                xf=1.0, yf=1.0)
b = PROBLEMS[{name!r}]()
st, h = create(b, {precision!r})
want = workspace(h)
lib.snac_plan_destroy(h)
arr, keep = snac._marshal_blocks(b)
n3 = sum(int(np.prod([q["hi"][a] - q["lo"][a] + 1 for a in range(3)])) for q in b)
f, p = np.zeros(n3), np.empty(n3)
o = snac._Options(snac._PREC[{precision!r}], 2, 2, 20, 40, 64, -1, 0.0, 0.0, 0, 0, 0, 0)
out = [st, want]
vcycles = n3 * (16 + (64 if {precision!r} == "fp64" else 40)) + (64 << 20)
for budget in (1 << 40, vcycles):
    eo = snac._EngineOptions(1, 8, budget, 0, 16)
    e, t = ctypes.c_void_p(), ctypes.c_int64()
    fake.fake_reset()
    before = fake.fake_used()
    r = [lib.snac_engine_create(ctypes.byref(e), ctypes.byref(eo)),
         lib.snac_engine_submit(e, len(b), arr, 2, ctypes.byref(o), f.ctypes.data, p.ctypes.data, 1e-10, ctypes.byref(t)),
         lib.snac_engine_wait(e, t, None, None)]
    s = snac._EngineStats()
    lib.snac_engine_get_stats(e, ctypes.byref(s))
    out.append([r, fake.fake_peak() - before, s.bytes_peak, any("k_resp" in l for l in launches())])
    lib.snac_engine_destroy(e)
""")
    st, want, wide, tight = out
    assert st == 0 and wide[0] == tight[0] == [0, 0, 0]
    assert wide[1] <= wide[2] and tight[1] <= tight[2] and want <= wide[2]
    pieces = name in ("thin", "L", "T")
    assert wide[3] == pieces and not tight[3]


@pytest.mark.parametrize("name", ["L", "L on chip"])
def test_equal_shifts_share_an_interface_system(name):
    """Wavenumbers q and n - q of a periodic z have one eigenvalue: n / 2 + 1 inverses are kept, not n."""
    out = fake_cuda.run(LAYOUTS + f"""
out = []
n, k = (160, 80) if {name!r} == "L" else (32, 16)
pivots = 3 * k * k if {name!r} == "L" else 0   # (kept with the plan off chip, shared likewise)
for nz in (32, 64):
    ws = []
    for walls in ("DNNN", "NNNN"):
        for z in (("P", "P"), ("N", "N")):
            st, h = create(problem(L(n // 2), n, n, nz=nz, z=z, walls=walls))
            ws.append(workspace(h))
    out.append([ws[1] - ws[0], ws[3] - ws[2]])
out = [out[1][i] - out[0][i] - (31 - 15) * 8 * (k * k + pivots) for i in range(2)]
""")
    assert all(x >= 0 for x in out)
