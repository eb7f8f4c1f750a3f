"""Stage (a) on the tensor cores, all callers, on the two grids it is built for: row tiles of 128
conduction bands (one short, one exact, one over), partial valence tiles, odd and even numbers of kept
z-frequencies, chunks that hold less than a row of pairs, and a conduction set of several blocks.
Against the library's FP64 mode, which shares the digit step and the contraction's kernel with the mode under
test and is itself held to the FP64 FFT kernel's pair elements contracted on DMMA.  Two-float stage (a) keeps 2e-13 and the
contraction at seven-slice accuracy, a five-slice expansion, 32 * 5 * 2^-45 = 5e-12 of the product of two
columns' largest magnitudes per pair: relative to the columns' norms below 2e-11 for these bands."""
import numpy as np
import pytest

import gwgen

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
TOL = 2e-11


@pytest.fixture(scope="module")
def gw():
    if not torch.cuda.is_available():
        pytest.fail("GPU tests need a CUDA device")
    import paper_2509_23018_gb300 as gw
    return gw


def dev(x):
    return torch.as_tensor(np.ascontiguousarray(x), device="cuda")


def rel(a, b):
    return float(torch.linalg.vector_norm(a - b) / torch.linalg.vector_norm(b))


SHAPES = [(40, 9, 127, 1500, 333, 8192), (40, 33, 256, 3000, 900, 4096), (40, 4, 129, 1500, 401, 8192),
          (48, 20, 300, 2500, 700, 2100), (48, 7, 500, 2000, 500, 400), (48, 3, 1100, 3000, 300, 8192)]


@pytest.mark.parametrize("n,nv,nc,ngpsi,ng,chunk", SHAPES)
def test_route_matches_fp64(gw, n, nv, nc, ngpsi, ng, chunk):
    p = gwgen.make_problem((n, n, n), nv, nc, ngpsi, ng, seed=n + nv)
    rng = np.random.default_rng(nc)
    W = dev(gwgen.hermitian(rng, ng))
    tan = [dev(rng.standard_normal(c.shape) + 1j * rng.standard_normal(c.shape)) * 1e-2 for c in (p.cv, p.cc)]
    tan += [dev(rng.standard_normal(len(e))) for e in (p.ev, p.ec)]
    basis = dev(np.linalg.qr(rng.standard_normal((ng, 24)) + 1j * rng.standard_normal((ng, 24)))[0])
    out = {}
    for mode, kw in (("fp64", dict(prec="fp64")), ("split", dict(prec="ozaki", nslices=7, mtxel="twofloat"))):
        h = gw.from_problem(p, pair_chunk=chunk, **kw)
        if mode == "split":
            assert h.streams(0) == 1
        else:  # other kernels from the bands on: the FFT pair kernel and the contraction of given elements
            dmma = h.contract(dev(p.ev), dev(p.ec), h.pair_elements(0, 0, nv * nc), [0.0, 3.0])
            assert rel(h.compute(0, [0.0, 3.0])[0], dmma) < 5e-15
        r = {"chi": h.compute(0, [0.0, 3.0])[0], "batch": h.compute_batch([0], [0.0, 3.0])[0],
             "sub": h.compute_subspace(0, basis, [1.0]), "real": h.compute_real(0, [4.0], 0.2),
             "jvp": h.jvp(0, [2.0], *tan)}
        r.update(zip(("dev", "dec", "dcv", "dcc"), h.adjoint(0, W)[1:]))
        h.keep_pair_elements(True)
        r["kept"] = h.compute(0, [0.0])[0]
        r["kept_sub"] = h.compute_subspace(0, basis, [1.0])
        h.sync()
        out[mode] = {k: v.clone() for k, v in r.items()}
        h.destroy()
    # the forward derivative and the real axis subtract contractions of larger magnitude
    loose = {"jvp": 5, "real": 5, "dev": 5, "dec": 5}
    bad = {k: rel(v, out["fp64"][k]) for k, v in out["split"].items() if rel(v, out["fp64"][k]) > TOL * loose.get(k, 1)}
    assert not bad


def test_route_yields_to_the_memory_budget(gw):
    """A budget without room for the route's buffers: the FFT pair kernel serves the call as before."""
    p = gwgen.make_problem((40, 40, 40), 8, 200, 1500, 300, seed=9)
    ref = gw.from_problem(p, prec="fp64").compute(0, [0.0])[0]
    # grids, pair elements and slices need about 0.25 GB; the route's slices and F 0.6 GB more
    h = gw.from_problem(p, prec="ozaki", nslices=7, mtxel="twofloat", mem_budget_bytes=500 << 20)
    assert rel(h.compute(0, [0.0])[0], ref) < TOL
    h.sync()
    assert h.device_bytes() <= 500 << 20


@pytest.mark.parametrize("op", ["jvp", "real", "sub", "adjoint", "chi", "chi1"])
def test_more_budget_never_fails(gw, op):
    """Budgets in steps of 80 MB through the range where the route's buffers begin to fit (slices 0.6 GB, F and
    cells more): once a call runs, it runs with every larger budget, and gives the same."""
    p = gwgen.make_problem((40, 40, 40), 12, 300, 3000, 900, seed=4)
    rng = np.random.default_rng(4)
    tan = [dev(rng.standard_normal(c.shape) + 1j * rng.standard_normal(c.shape)) * 1e-2 for c in (p.cv, p.cc)]
    tan += [dev(rng.standard_normal(len(e))) for e in (p.ev, p.ec)]
    basis = dev(np.linalg.qr(rng.standard_normal((900, 40)) + 1j * rng.standard_normal((900, 40)))[0])
    W = dev(gwgen.hermitian(rng, 900))
    run = {"jvp": lambda h: h.jvp(0, [0.0, 2.0], *tan), "real": lambda h: h.compute_real(0, [1.0, 4.0, 8.0], 0.1),
           "sub": lambda h: h.compute_subspace(0, basis, [0.0]), "adjoint": lambda h: h.adjoint(0, W)[4],
           "chi": lambda h: h.compute(0, [0.0, 1.0])[0], "chi1": lambda h: h.compute(0, [0.0])[0]}[op]
    kw = dict(prec="ozaki", nslices=7, mtxel="twofloat")
    ref, ran = run(gw.from_problem(p, **kw)), []
    for step in range(30):
        budget = int(0.4e9) + step * (80 << 20)
        try:
            h = gw.from_problem(p, mem_budget_bytes=budget, **kw)
            for _ in range(2):  # the second call finds what the first has left
                assert rel(run(h), ref) < 5 * TOL
            h.sync()
            assert h.device_bytes() <= budget
            ran.append(True)
        except gw.GwError as e:
            assert "OOM" in str(e)
            ran.append(False)
    assert ran[-1] and ran == sorted(ran)


def test_eight_slices_keep_the_fft_kernel_elsewhere(gw):
    """At eight slices the pair elements' own error would show: other calls than chi on 48^3 keep the FFT
    kernel and stay within its error (bound of the six-slice expansion: 32 * 6 * 2^-54 = 1e-14 a pair)."""
    p = gwgen.make_problem((40, 40, 40), 8, 200, 1500, 300, seed=9)
    ref = gw.from_problem(p, prec="fp64").compute(0, [0.0])[0]
    h = gw.from_problem(p, prec="ozaki", nslices=8, mtxel="twofloat")
    assert rel(h.compute(0, [0.0])[0], ref) < 4e-14
    h.sync()


@pytest.mark.parametrize("chunk", [500, 8192])
def test_overlap_where_the_route_declines(gw, chunk):
    """40^3 at eight slices keeps the FFT kernel, and with it the contraction beside it on a second stream: the same
    bits as on one stream; and a call on one stream where a budget has no room for the second slice buffer."""
    p = gwgen.make_problem((40, 40, 40), 8, 200, 1500, 300, seed=9)
    kw = dict(prec="ozaki", nslices=8, mtxel="twofloat", pair_chunk=chunk)
    one, two = gw.from_problem(p, single_stream=True, **kw), gw.from_problem(p, **kw)
    assert (one.streams(0), two.streams(0)) == (1, 2)
    want = one.compute(0, [0.0])[0]
    one.sync()
    assert torch.equal(two.compute(0, [0.0])[0], want)
    two.sync()
    used = one.device_bytes()
    for over in (1 << 20, 6 << 20, 64 << 20):
        h = gw.from_problem(p, mem_budget_bytes=used + over, **kw)
        assert rel(h.compute(0, [0.0])[0], want) < 4e-14  # tiles in parts may be whole ones here
        h.sync()
        assert h.device_bytes() <= used + over


@pytest.mark.parametrize("op", ["chi", "batch", "real"])
@pytest.mark.parametrize("n,nv,nc,chunk,route", [(48, 40, 2, 8192, False), (48, 8, 128, 8192, True), (40, 40, 2, 8192, False),
                                                 (72, 13, 1, 8192, False), (72, 8, 128, 8192, True)])
def test_small_calls_take_the_faster_kernel(gw, n, nv, nc, chunk, route, op):
    """Few conduction bands fill little of a tile of 128 rows, and each tile of valence bands costs as much as a
    full one: those calls keep the FFT kernel, and both give the same."""
    p = gwgen.make_problem((n, n, n), nv, nc, 5 * n * n // 6, n * n // 3, seed=n + nc)
    run = {"chi": lambda h: h.compute(0, [0.0, 2.0])[0], "batch": lambda h: h.compute_batch([0], [0.0, 2.0])[0],
           "real": lambda h: h.compute_real(0, [1.0], 0.1)}[op]
    h = gw.from_problem(p, prec="ozaki", nslices=7, mtxel="twofloat", pair_chunk=chunk, single_stream=True)
    got = run(h)
    h.sync()
    if op != "batch":  # (captured: no times)
        h.set_timing(True)
        run(h)
        h.sync()
        assert ("zdft" in h.timing(reset=True)) == route
    assert rel(got, run(gw.from_problem(p, prec="fp64"))) < 5 * TOL


@pytest.mark.parametrize("nv,nc", [(2, 1), (2, 32), (16, 30)])
def test_sphere_of_few_vectors_takes_the_faster_kernel(gw, nv, nc):
    """The FFT kernel takes less time the fewer frequencies a sphere keeps along the last axis; 27 vectors on 48^3 stay
    on it, and match FP64."""
    p = gwgen.make_problem((48, 48, 48), nv, nc, 2000, 27, seed=nc)
    h = gw.from_problem(p, prec="ozaki", nslices=7, mtxel="twofloat")
    h.set_timing(True)
    got = h.compute(0, [0.0, 2.0])[0]
    h.sync()
    assert "zdft" not in h.timing(reset=True)
    assert rel(got, gw.from_problem(p, prec="fp64").compute(0, [0.0, 2.0])[0]) < 5 * TOL


@pytest.mark.parametrize("prec,mtxel", [("ozaki", "twofloat"), ("fp64", "fp64")])
def test_batch_of_chunks_below_a_tile(gw, prec, mtxel):
    """A batch's blocks follow the pair chunk, its FFT launch does not: 40 x 7 bands in chunks of 100 pairs stay on
    the FFT kernel, and match the streamed call."""
    p = gwgen.make_problem((48, 48, 48), 40, 7, 2000, 400, seed=3)
    h = gw.from_problem(p, prec=prec, nslices=7, mtxel=mtxel, pair_chunk=100)
    a, b = h.compute_batch([0], [0.0, 2.0])[0], h.compute(0, [0.0, 2.0])[0]
    h.sync()
    assert rel(a, b) < (TOL if prec == "ozaki" else 5e-15)
