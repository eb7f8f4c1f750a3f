"""FP64 stage (a) with the last axis on the tensor cores: pair elements' contraction on grids of every
length its kernels serve, lines that do not fill their stages, odd first axes, partial row and valence
tiles, one row tile and several, chunks below a row of pairs.  Against the FP64 FFT kernel's pair elements
(gw_chi0_pair_elements) contracted by torch in FP64; both carry a few roundings of 2^-53 per element.
Entries that are not finite, and scales beyond 2^+-390, go to the FFT kernel."""
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
