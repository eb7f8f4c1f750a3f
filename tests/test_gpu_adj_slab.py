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
                                              (40, 6, 50, 900, 300), (48, 7, 33, 900, 250),
                                              (40, 1, 30, 900, 300), (40, 4, 30, 900, 300), (40, 5, 30, 900, 300),
                                              (48, 3, 33, 900, 250)])
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


@pytest.mark.parametrize("m", [(0, 34, 17), (1, 25, 17)])
def test_wide_spheres(gw, m):
    """Boxes of G on 72^3 whose (k1, k2) cells (2415 and 1785) go beyond and up to what a slab block's shared memory
    holds: gradients against the oracle's adjoint, as the runtime-shape kernel gives them."""
    import oracle
    axes = lambda k: np.stack(np.meshgrid(*[np.arange(-x, x + 1) for x in k], indexing="ij"), -1).reshape(-1, 3)  # noqa: E731
    gchi, gpsi = axes(m).astype(np.int32), axes((1, 1, 0)).astype(np.int32)
    rng = np.random.default_rng(m[1])
    q = np.linalg.qr(rng.standard_normal((9, 9)) + 1j * rng.standard_normal((9, 9)))[0]
    cv, cc, ev, ec = q[:1], q[1:4], np.array([-1.0]), np.array([1.0, 2.0, 4.0])
    W = gwgen.hermitian(rng, len(gchi))
    dev = lambda x: torch.as_tensor(np.ascontiguousarray(x), device="cuda")  # noqa: E731
    h = gw.Chi0((72, 72, 72), prec="ozaki", nslices=7, mtxel="twofloat")
    h.set_bands(0, 1, dev(gpsi), dev(cc), dev(ec))
    h.set_bands(0, 0, dev(gpsi), dev(cv), dev(ev))
    h.set_gsphere(0, dev(gchi))
    got = h.adjoint(0, dev(W), omega=1.0)
    h.sync()
    h.destroy()
    want = oracle.adjoint(gpsi, cv, ev, gpsi, cc, ec, gchi, W, 1.0)
    for a, b in zip(got[1:], want[1:]):
        assert np.linalg.norm(a.cpu().numpy() - b) < 1e-10 * np.linalg.norm(b)
