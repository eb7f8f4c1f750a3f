"""The dielectric inverse, whose early steps take three or four slices where their error allows: matrices
near the identity (few steps) to a bound of 600 (many), and the handle's own accuracy below, at and above
those.  Against a dense FP64 inverse; the last two steps run with six slices, 2^-54 of the rows' and columns'
largest entries a product, times the condition number of at most 600: 1e-10 of the inverse's norm."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,scale,nslices", [(40, 1e-3, 7), (150, 0.5, 7), (300, 5.0, 7), (300, 60.0, 7), (300, 5.0, 3),
                                             (300, 5.0, 5), (300, 60.0, 8), (700, 300.0, 6)])
def test_inverse_matches_dense(n, scale, nslices):
    if not torch.cuda.is_available():
        pytest.fail("GPU tests need a CUDA device")
    import paper_2509_23018_gb300 as gw
    rng = np.random.default_rng(n)
    a = rng.standard_normal((n, 2 * n)) + 1j * rng.standard_normal((n, 2 * n))
    chi = torch.as_tensor(-scale / (4.0 * n) * (a @ a.conj().T), device="cuda")
    v = torch.as_tensor(1.0 / (1.0 + np.arange(n) / n), device="cuda")
    h = gw.Chi0((24, 24, 24), prec="ozaki", nslices=nslices, mtxel="twofloat")
    got = h.epsilon_inverse(chi[None], v)[0]
    h.sync()
    ref = torch.linalg.inv(torch.eye(n, dtype=torch.complex128, device="cuda") - v[:, None] * chi)
    assert float(torch.linalg.vector_norm(got - ref) / torch.linalg.vector_norm(ref)) < 1e-10
