"""Stage (a) on the tensor cores on grids other than 40^3 and 48^3: every axis length its middle- and
first-axis kernels are built for, odd first axes (half a slab pair at the end), last axes that do not fill
their stages of eight points, tiles of 96 columns (60 to 72 points; 72 loads its lines in halves), odd
numbers of kept frequencies, partial row and valence tiles, chunks of less than a row of pairs.  Against
the library's FP64 mode (1e-15), and the route's own kernels have run.  Tolerance of
the route's error at seven slices, a five-slice expansion: 32 * 5 * 2^-45 = 5e-12 of the product of two
columns' largest magnitudes per pair, relative to the columns' norms below 2e-11 for these bands."""
import gwgen
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
TOL = 2e-11


@pytest.fixture(scope="module")
def gw():
    if not torch.cuda.is_available():
        pytest.fail("GPU tests need a CUDA device")
    import paper_2509_23018_gb300 as gw
    return gw


SHAPES = [((30, 36, 40), 13, 147, 700, 333, 8192), ((25, 32, 27), 9, 150, 500, 200, 700),
          ((20, 45, 25), 7, 260, 400, 150, 130), ((27, 24, 64), 8, 129, 500, 257, 8192),
          ((36, 20, 45), 5, 200, 400, 200, 8192), ((64, 25, 30), 6, 128, 500, 180, 500),
          ((45, 50, 54), 6, 131, 1500, 700, 8192), ((54, 27, 50), 6, 140, 700, 300, 8192),
          ((32, 60, 36), 11, 200, 900, 500, 8192), ((50, 64, 60), 4, 130, 2000, 1100, 300),
          ((60, 54, 72), 5, 129, 2500, 1500, 8192), ((48, 40, 24), 6, 150, 600, 250, 8192),
          ((24, 30, 32), 12, 140, 600, 250, 8192), ((40, 48, 48), 9, 130, 1500, 600, 8192),
          ((72, 72, 72), 9, 140, 8000, 6000, 8192), ((36, 36, 36), 11, 130, 900, 450, 8192)]


@pytest.mark.parametrize("grid,nv,nc,ngpsi,ng,chunk", SHAPES)
def test_grids_match_fp64(gw, grid, nv, nc, ngpsi, ng, chunk):
    p = gwgen.make_problem(grid, nv, nc, ngpsi, ng, seed=sum(grid))
    out = {}
    for mode, kw in (("fp64", dict(prec="fp64")), ("split", dict(prec="ozaki", nslices=7, mtxel="twofloat"))):
        h = gw.from_problem(p, pair_chunk=chunk, **kw)
        h.set_timing(True)
        r = [h.compute(0, [0.0, 3.0])[0]]
        h.sync()
        ran = set(h.timing(reset=True))
        assert mode == "fp64" or "zdft" in ran, ran
        h.set_timing(False)
        r.append(h.compute_batch([0], [2.0])[0])
        h.keep_pair_elements(True)
        r.append(h.compute(0, [0.0])[0])
        h.sync()
        out[mode] = [x.clone() for x in r]
        h.destroy()
    for a, b in zip(out["split"], out["fp64"]):
        assert float(torch.linalg.vector_norm(a - b) / torch.linalg.vector_norm(b)) < TOL
