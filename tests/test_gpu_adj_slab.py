"""The back-projection in cells and slabs on each cubic grid it is built for, spheres of several batches
of cells and of less than one, against the FP64 mode's gradients (another kernel); and a sphere with
more columns than the slab's buffers hold, which stays on the runtime-shape kernel; one to seven
valence rows for the products that read each grid once (up to six).  Two-float steps carry
2^-46 each, the seven-slice products 5e-12 of the columns' norms: 1e-10 of the gradients' norms."""
import gwgen
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gw():
    if not torch.cuda.is_available():
        pytest.fail("GPU tests need a CUDA device")
    import paper_2509_23018_gb300 as gw
    return gw


@pytest.mark.parametrize("n,nv,nc,ngpsi,ng", [(24, 3, 40, 60, 19), (24, 2, 30, 60, 1000), (40, 3, 37, 900, 700),
                                              (48, 2, 40, 2000, 1500), (72, 1, 30, 3000, 2500), (24, 2, 30, 19, 2000),
                                              (40, 6, 50, 900, 300), (48, 7, 33, 900, 250)])
def test_gradients_match_fp64(gw, n, nv, nc, ngpsi, ng):
    p = gwgen.make_problem((n, n, n), nv, nc if nc + nv <= ngpsi else ngpsi - nv, ngpsi, ng, seed=n + ng)
    W = torch.as_tensor(gwgen.hermitian(np.random.default_rng(2), ng), device="cuda")
    out = []
    for kw in (dict(prec="fp64"), dict(prec="ozaki", nslices=7, mtxel="twofloat")):
        h = gw.from_problem(p, **kw)
        out.append([x.clone() for x in h.adjoint(0, W, omega=1.0)[1:]])
        h.sync()
        h.destroy()
    for a, b in zip(out[1], out[0]):
        assert float(torch.linalg.vector_norm(a - b) / torch.linalg.vector_norm(b)) < 1e-10
