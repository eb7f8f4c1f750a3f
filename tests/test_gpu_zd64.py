"""FP64 stage (a) with the last axis on the tensor cores: pair elements' contraction on grids of every
length its kernels serve, lines that do not fill their stages, odd first axes, partial row and valence
tiles, one row tile and several, chunks below a row of pairs.  Against the FP64 FFT kernel's pair elements
(gw_chi0_pair_elements) contracted by torch in FP64; both carry a few roundings of 2^-53 per element.
Entries that are not finite, and scales beyond 2^+-390, go to the FFT kernel."""
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


SHAPES = [((24, 24, 24), 16, 64, 300, 200, 8192), ((25, 32, 27), 9, 150, 500, 200, 700),
          ((20, 45, 25), 7, 260, 400, 150, 130), ((27, 24, 50), 8, 129, 500, 257, 8192),
          ((36, 20, 45), 5, 200, 400, 200, 8192), ((64, 25, 30), 6, 128, 500, 180, 500),
          ((45, 50, 54), 6, 131, 1500, 700, 8192), ((32, 60, 36), 11, 200, 900, 500, 8192),
          ((72, 54, 32), 4, 140, 900, 450, 8192), ((48, 48, 48), 7, 300, 4000, 1400, 8192),
          ((30, 40, 48), 3, 600, 700, 250, 8192)]


@pytest.mark.parametrize("grid,nv,nc,ngpsi,ng,chunk", SHAPES)
def test_chi_matches_the_fft_kernel(gw, grid, nv, nc, ngpsi, ng, chunk):
    p = gwgen.make_problem(grid, nv, nc, ngpsi, ng, seed=sum(grid))
    h = gw.from_problem(p, prec="fp64", pair_chunk=chunk)
    h.set_timing(True)
    om = [0.0, 2.0]
    chi = h.compute(0, om)[0]
    h.sync()
    assert "zdft" in h.timing(reset=True)
    M = h.pair_elements(0, 0, nv * nc)
    batch = h.compute_batch([0], om)[0]
    h.sync()
    x = (torch.as_tensor(p.ev)[:, None] - torch.as_tensor(p.ec)[None, :]).reshape(-1, 1).cuda()
    for got in (chi, batch):
        for i, w in enumerate(om):
            ref = M.mH @ (4.0 * x / (x * x + w * w) * M)
            assert float(torch.linalg.vector_norm(got[i] - ref) / torch.linalg.vector_norm(ref)) < TOL
    h.destroy()


@pytest.mark.parametrize("scale", [2.0 ** -420, 2.0 ** 100, float("nan"), float("inf")])
def test_what_slices_cannot_hold_goes_to_the_fft_kernel(gw, scale):
    p = gwgen.make_problem((24, 24, 24), 5, 130, 300, 200, seed=3)
    q = gwgen.make_problem((24, 24, 24), 5, 130, 300, 200, seed=3)
    if np.isfinite(scale):
        q.cv, q.cc = q.cv * scale, q.cc / scale
    else:
        q.cc[7, 3] = scale
    chi = gw.from_problem(q, prec="fp64").compute(0, [0.0])[0]
    if np.isfinite(scale):
        ref = gw.from_problem(p, prec="fp64").compute(0, [0.0])[0]
        assert float(torch.linalg.vector_norm(chi - ref) / torch.linalg.vector_norm(ref)) < TOL
    else:
        assert bool(torch.isnan(torch.view_as_real(chi)).any(-1).all())


def digits_value(d):
    """The value below 1 whose balanced base-512 digits, relative to a largest entry in [1/2, 1), are d, 0, 0, ..."""
    return float(sum(Fraction(v) * Fraction(512) ** (6 - i) for i, v in enumerate(d)) / Fraction(2) ** 61)


@pytest.mark.parametrize("grid", [(32, 24, 32), (24, 32, 40), (48, 48, 48), (25, 20, 50), (24, 24, 54)])
@pytest.mark.parametrize("low", [243, 200])
def test_lines_of_coherent_digits(gw, grid, low):
    """Nearly constant bands whose leading digits lie near their largest with one sign, and whose next ones vary along
    the last axis: the sums over a line of the products i + j = 3 and 4 come close to their largest.  The valence
    band is constant, v (1 + i), the conduction bands c (1 + i) and a wave of 2^-32 along z; up to 30 pairs, whose
    contraction stays on DMMA, against the exact sum."""
    rng = np.random.default_rng(sum(grid) + low)
    nb = 16
    g = np.stack(np.meshgrid([0, 1, -1], [0, 1, -1], [0, 1, -1], indexing="ij"), -1).reshape(-1, 3).astype(np.int32)
    cc, cv = np.zeros((nb, 27), complex), np.zeros((1, 27), complex)
    cv[0, 0] = digits_value([63, 255, 255, 254]) * (1 + 1j)
    cc[:, 0] = digits_value([127, 255, 255, low]) * (1 + 1j)
    cc[:, 1:3] = 2.0 ** -32 * (rng.uniform(-1, 1, (nb, 2)) + 1j * rng.uniform(-1, 1, (nb, 2)))
    gchi = np.array([[0, 0, 0], [0, 0, 1], [0, 0, -1], [0, 1, 0], [1, 0, 0]], np.int32)
    dev = lambda x: torch.as_tensor(np.ascontiguousarray(x), device="cuda")  # noqa: E731
    h = gw.Chi0(grid, prec="fp64")
    h.set_bands(0, 1, dev(g), dev(cc), dev(np.full(nb, 2.0)))
    h.set_bands(0, 0, dev(g), dev(cv), dev(np.full(1, -2.0)))
    h.set_gsphere(0, dev(gchi))
    h.set_timing(True)
    chi = h.compute(0, [0.0])[0][0].cpu().numpy()
    h.sync()
    assert "zdft" in h.timing(reset=True)
    h.destroy()
    # M(0) = conj(c_v(0)) c_c(0): the wave has no overlap with the valence band
    frac = lambda z: (Fraction(float(z.real)), Fraction(float(z.imag)))  # noqa: E731
    (a, b), want = frac(cv[0, 0]), Fraction(0)
    for z in cc[:, 0]:
        x, y = frac(z)
        want -= (a * x + b * y) ** 2 + (a * y - b * x) ** 2
    assert abs((Fraction(float(chi[0, 0].real)) - want) / want) < TOL
