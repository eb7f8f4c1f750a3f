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


@pytest.mark.parametrize("kind", ["uniform", "phases", "random"])
@pytest.mark.parametrize("n,bulk,strength,nslices", [(600, 0.1, 300.0, 7), (1500, 0.1, 100.0, 7), (1500, 0.1, 1e4, 7),
                                                     (2000, 0.0, 1e3, 7), (1500, 0.1, 1e4, 3)])
def test_strong_spread_mode(n, bulk, strength, nslices, kind):
    """A bulk near the identity and one strong mode spread over all G, equal entries among them (every digit of
    a row the same): steps that start just below a residual of 1, where a product's error may undo what the
    step gains (and does with a handle of three slices, whose early steps are taken again).  Bound: the last steps' rounding, 8 n 2^-54 (the model of eps_step_slices for six slices) times
    the condition number."""
    if not torch.cuda.is_available():
        pytest.fail("GPU tests need a CUDA device")
    import paper_2509_23018_gb300 as gw
    rng = np.random.default_rng(n)
    a = rng.standard_normal((n, n)) + 1j * rng.standard_normal((n, n))
    u = {"uniform": np.ones(n), "phases": np.exp(2j * np.pi * rng.random(n)), "random": a[:, 0].copy()}[kind]
    u = u / np.linalg.norm(u)
    chi = torch.as_tensor(-bulk / (2.0 * n) * (a @ a.conj().T) - strength * np.outer(u, u.conj()), device="cuda")
    chi = 0.5 * (chi + chi.mH)
    v = torch.ones(n, dtype=torch.float64, device="cuda")
    h = gw.Chi0((24, 24, 24), prec="ozaki", nslices=nslices, mtxel="twofloat")
    got = h.epsilon_inverse(chi[None], v)[0]
    h.sync()
    ref = torch.linalg.inv(torch.eye(n, dtype=torch.complex128, device="cuda") - chi)
    tol = 8 * n * 2.0 ** -54 * (1.0 + strength)
    assert float(torch.linalg.vector_norm(got - ref) / torch.linalg.vector_norm(ref)) < tol
