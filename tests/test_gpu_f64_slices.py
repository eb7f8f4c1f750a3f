"""FP64 contraction by slices: spheres around its tiles of 128 columns, pair counts that leave K-steps of 64
and K blocks of 1024 short, several frequencies, split tiles, and the chunks that it leaves to the DMMA
kernel (entries that are not finite, scales beyond 2^+-390).  Against the same contraction of the library's
own pair elements in torch's FP64: both round a few times per entry, 2^-53 of the columns' norms each."""
from fractions import Fraction

import gwgen
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
TOL = 5e-15


@pytest.fixture(scope="module")
def gw():
    if not torch.cuda.is_available():
        pytest.fail("GPU tests need a CUDA device")
    import paper_2509_23018_gb300 as gw
    return gw


def problem(nv, nc, ng, scale=1.0):
    p = gwgen.make_problem((32, 32, 32), nv, nc, 1500, ng, seed=nv + nc + ng)
    p.cv, p.cc = p.cv * scale, p.cc * scale
    return p


def reference(p, M, omega):
    x = (torch.as_tensor(p.ev)[:, None] - torch.as_tensor(p.ec)[None, :]).reshape(-1, 1).cuda()
    return M.mH @ (4.0 * x / (x * x + omega * omega) * M)


SHAPES = [(5, 130, 200, 8192), (9, 227, 128, 8192), (16, 129, 129, 2000), (31, 67, 255, 1025), (7, 293, 300, 8192),
          (3, 1000, 384, 8192), (64, 300, 257, 19200)]


@pytest.mark.parametrize("nv,nc,ng,chunk", SHAPES)
def test_chi_matches_fp64(gw, nv, nc, ng, chunk):
    p = problem(nv, nc, ng)
    h = gw.from_problem(p, prec="fp64", pair_chunk=chunk)
    om = [0.0, 3.0]
    h.set_timing(True)
    chi = h.compute(0, om)[0]
    h.sync()
    assert "oz_split" in h.timing(reset=True)
    M = h.pair_elements(0, 0, nv * nc)
    again = h.compute(0, om)[0]
    for i, w in enumerate(om):
        ref = reference(p, M, w)
        assert float(torch.linalg.vector_norm(chi[i] - ref) / torch.linalg.vector_norm(ref)) < TOL
        d = torch.linalg.diagonal(ref).abs().sqrt()   # entry by entry, of the columns' norms
        assert float(((chi[i] - ref).abs() / (d[:, None] * d[None, :])).max()) < TOL
    assert torch.equal(chi, again)
    h.sync()
    h.destroy()


def digits_value(d):
    """The value in [1, 2) whose seven balanced base-512 digits, relative to a largest entry in [1, 2), are d."""
    return float(sum(Fraction(v) * Fraction(512) ** (6 - i) for i, v in enumerate(d)) / Fraction(2) ** 61)


COHERENT = [[(127, 127), (255, 255), (200, 255)], [(127, 127), (254, 255)], [(127, 127), (255, 255), (255, 255), (200, 255)],
            [(127, 127)] + [(255, 255)] * 3 + [(200, 255)] * 2, [(120, 127)] + [(230, 255)] * 6, [(64, 64)] + [(-256, -230)] * 6]


@pytest.mark.parametrize("nc", [4096, 700])
@pytest.mark.parametrize("ranges", COHERENT)
def test_sums_of_coherent_digits(gw, ranges, nc):
    """Pair elements that nearly coincide, so that the digits of a slice have one sign over all pairs and the
    FP32 sums of a slice group come close to their largest: one plane wave per band, M(0) = c, Delta = -1.
    chi(0, 0) = -sum c^2, summed exactly."""
    rng = np.random.default_rng(len(ranges) + nc)
    rows = [ranges[i] if i < len(ranges) else (-255, 255) for i in range(7)]
    c = np.array([digits_value([int(rng.integers(lo, hi + 1)) for lo, hi in rows]) for _ in range(nc)])
    g = np.stack(np.meshgrid([0, 1, -1], [0, 1, -1], [0, 1, -1], indexing="ij"), -1).reshape(-1, 3).astype(np.int32)
    coeff = lambda x: torch.as_tensor(np.outer(x, np.eye(27)[0]).astype(complex), device="cuda")  # noqa: E731
    vec = lambda x, n: torch.full((n,), x, dtype=torch.float64, device="cuda")  # noqa: E731
    h = gw.Chi0((32, 32, 32), prec="fp64")
    gd = torch.as_tensor(g, device="cuda")
    h.set_bands(0, 1, gd, coeff(c), vec(2.0, nc))
    h.set_bands(0, 0, gd, coeff(np.ones(1)), vec(-2.0, 1))
    h.set_gsphere(0, gd)
    chi = h.compute(0, [0.0])[0][0].cpu().numpy()
    h.sync()
    h.destroy()
    want = -sum(Fraction(x) ** 2 for x in c)
    assert abs((Fraction(float(chi[0, 0].real)) - want) / want) < TOL


@pytest.mark.parametrize("scale", [2.0 ** -200, 2.0 ** 210, float("nan"), float("inf")])
def test_what_slices_cannot_hold_goes_to_the_dmma_kernel(gw, scale):
    p = problem(5, 130, 200)
    ref = gw.from_problem(p, prec="fp64").compute(0, [0.0])[0]
    if np.isfinite(scale):
        q = problem(5, 130, 200, scale)
    else:
        q = problem(5, 130, 200)
        q.cc[7, 3] = scale
    chi = gw.from_problem(q, prec="fp64").compute(0, [0.0])[0]
    if np.isfinite(scale):
        back = chi / scale ** 2 / scale ** 2
        assert float(torch.linalg.vector_norm(back - ref) / torch.linalg.vector_norm(ref)) < TOL
    else:
        assert bool(torch.isnan(torch.view_as_real(chi)).any(-1).all())


def test_slices_make_room_for_what_a_call_needs(gw):
    """A memory budget that holds the slices of a small sphere or the pair elements of a large one: both
    calls run, in either order."""
    p, large = problem(16, 512, 125), gwgen.make_problem((32, 32, 32), 2, 3, 1500, 1000, seed=1).gchi
    dev = lambda x: torch.as_tensor(np.ascontiguousarray(x), device="cuda")  # noqa: E731

    def load(**kw):
        h = gw.Chi0(p.grid, nq=2, prec="fp64", pair_chunk=8192, **kw)
        h.set_bands(0, 1, dev(p.gpsi), dev(p.cc), dev(p.ec))
        for iq, g in ((0, p.gchi), (1, large)):
            h.set_bands(iq, 0, dev(p.gpsi), dev(p.cv), dev(p.ev))
            h.set_gsphere(iq, dev(g))
        return h

    free = load()
    budget = free.device_bytes() + 16 * 8192 * 1000 + (8 << 20)
    h = load(mem_budget_bytes=budget)
    h.set_timing(True)
    for iq in (0, 1, 0, 1):
        chi = h.compute([iq], [0.0])[0]
        h.sync()
        ran = "oz_split" in h.timing(reset=True)
        assert not ran if iq else True
        ref = free.compute([iq], [0.0])[0]
        assert float(torch.linalg.vector_norm(chi - ref) / torch.linalg.vector_norm(ref)) < TOL
        assert h.device_bytes() <= budget
        if (iq, ran) == (0, True):
            seen = True
    assert seen


@pytest.mark.parametrize("nv,nc,ng,nw,sliced", [(8, 7, 40, 9, False), (4, 8, 40, 1, True), (8, 7, 40, 1, True),
                                                (16, 64, 300, 9, True), (3, 30, 300, 9, False), (8, 127, 7, 9, False), (13, 129, 40, 27, False),
                                                (16, 512, 200, 9, True)])
def test_few_pairs_at_many_frequencies_stay_on_dmma(gw, nv, nc, ng, nw, sliced):
    """The slices cost a few launches a frequency, the DMMA kernel one for all: which of them runs, and the result."""
    p = problem(nv, nc, ng)
    h = gw.from_problem(p, prec="fp64", pair_chunk=100 if ng == 7 else 8192)
    om = [2.0 * k for k in range(nw)]
    h.set_timing(True)
    chi = h.compute(0, om)[0]
    h.sync()
    assert ("oz_split" in h.timing(reset=True)) == sliced
    M = h.pair_elements(0, 0, nv * nc)
    for i, w in enumerate(om):
        ref = reference(p, M, w)
        assert float(torch.linalg.vector_norm(chi[i] - ref) / torch.linalg.vector_norm(ref)) < TOL
    h.destroy()
