"""The split contraction and the general split product at the edges of their tiles (128 complex rows
and columns per pair of CTAs), K-steps (64 pairs), segments (256, 512 and 1024 pairs) and K parts,
entry by entry within the bound of the split itself.

With s nine-bit slices of x = 2^E u, |u| < 1/2: a slice sum is off by at most 2^(E - 9 s) (half a unit
of its last digit), a dropped product (i + k > s + 1) is at most 2^(E + E' + 2 - 9 (s + 2)) 2^16, and
there are s - 1 of them on the first dropped diagonal (the further ones are 2^-9 of it).  With 2^E at
most four times the largest magnitude, and two real products per part of a complex entry:
|error| <= 2 P s 2^(E + E' - 9 s) <= 32 P s 2^(-9 s) max|x| max|x'|."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SLICES = {3: 3, 4: 3, 5: 4, 6: 5, 7: 5, 8: 6}  # nine-bit slices for the requested accuracy


@pytest.fixture(scope="module")
def gw():
    if not torch.cuda.is_available():
        pytest.fail("GPU tests need a CUDA device")
    import paper_2509_23018_gb300 as gw
    return gw


def dev(x):
    return torch.as_tensor(np.ascontiguousarray(x), device="cuda")


def parts_max(a, axis):
    return np.maximum(np.abs(a.real), np.abs(a.imag)).max(axis=axis)


def bound(K, nslices, left, right):
    s = SLICES[nslices]
    return 32.0 * K * s * 2.0 ** (-9 * s) * np.outer(left, right) + 1e-15 * K * np.outer(left, right)


def contract(gw, M, nslices, **kw):
    """chi of M with Delta = -1 for every pair: -M^H M."""
    P = M.shape[0]
    h = gw.Chi0((8, 8, 8), prec="ozaki", nslices=nslices, **kw)
    chi = h.contract(dev(np.full(1, -2.0)), dev(np.full(P, 2.0)), dev(M), [0.0]).cpu().numpy()[0]
    h.sync()
    h.destroy()
    return chi


@pytest.mark.parametrize("ng,P,nslices", [(1, 1, 7), (63, 64, 7), (64, 65, 3), (65, 255, 7), (127, 256, 5),
                                          (128, 257, 7), (129, 511, 8), (255, 513, 4), (256, 1023, 6),
                                          (257, 1025, 7), (385, 4099, 7), (1300, 1537, 7)])
def test_contraction_edges(gw, ng, P, nslices):
    rng = np.random.default_rng(ng * 10007 + P)
    M = rng.standard_normal((P, ng)) + 1j * rng.standard_normal((P, ng))
    M *= 10.0 ** rng.uniform(-6, 6, ng)[None, :]  # columns of very different scales
    chi = contract(gw, M, nslices)
    assert np.array_equal(chi, chi.conj().T)
    mx = parts_max(M, 0)
    assert (np.abs(chi + M.conj().T @ M) <= np.sqrt(2.0) * bound(P, nslices, mx, mx)).all()


@pytest.mark.parametrize("value", [1.0 + 1.0j, 1.0 - 2.0 ** -20 + 0.5j, 4.0 - 2.0 ** -30 - 3.999j])
def test_contraction_largest_sums(gw, value):
    """Every pair carries the same value, so every digit of a column has one sign and every slice group
    reaches its largest sum.  t = 2 and 3 are exact then; a t = 4 segment of 256 pairs may round by a
    unit (2^-34 of the scale squared) in each of its 48 MMA steps, 2^-28 of 2^12 at most per pair part,
    and t >= 5 by less: 2^-34 of the sum covers them."""
    P, ng = 8192, 130
    chi = contract(gw, np.full((P, ng), value), 7)
    want = -P * abs(value) ** 2
    assert np.abs(chi - want).max() <= (2.0 ** -34 + 32 * 5 * 2.0 ** -45) * abs(want) * 2


@pytest.mark.parametrize("rows,cols,K,nslices", [(1, 1, 1, 7), (63, 127, 65, 7), (130, 128, 129, 6), (257, 129, 300, 7),
                                                 (64, 260, 1025, 8)])
def test_general_product_edges(gw, rows, cols, K, nslices):
    """Y = A B through the off-diagonal self-energy's two products: one band, one energy and a
    plasmon-pole matrix P = A0 that the call forms from its residues (v = 1, wt = i, E = E_n):
    sigma = conj(M) P M^T, with P = Omega^2 / (2 wt (-wt)) = Omega^2 / 2."""
    n = max(cols, K)
    rng = np.random.default_rng(rows + 1000 * cols + K)
    M = rng.standard_normal((1, rows, n)) + 1j * rng.standard_normal((1, rows, n))
    O2 = rng.standard_normal((n, n)) + 1j * rng.standard_normal((n, n))
    h = gw.Chi0((8, 8, 8), prec="ozaki", nslices=nslices)
    got = h.sigma_gpp(dev(M), [1.0], 0, dev(O2), dev(np.full((n, n), 1j)), dev(np.ones(n)), [1.0])
    got = got.cpu().numpy()[0]
    h.sync()
    h.destroy()
    Pm = O2 / 2.0
    X = M[0].conj() @ Pm
    # the prep. step holds P to 2^-43 of a row's largest part (two-float arithmetic)
    e1 = bound(n, nslices, parts_max(M[0], 1), parts_max(Pm, 0)) + n * 2.0 ** -42 * np.outer(
        parts_max(M[0], 1), parts_max(Pm, 0))
    e2 = bound(n, nslices, parts_max(X, 1), parts_max(M[0], 1))
    tol = np.sqrt(2.0) * e2 + 2.0 * e1 @ np.abs(M[0]).T
    assert (np.abs(got - X @ M[0].T) <= tol).all()
