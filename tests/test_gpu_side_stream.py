"""A handle used on a stream of its own while the default stream is busy: what the library clears or
uploads for itself has to be ordered with the handle's stream, not with the default one.  The default stream
copies for several times what the call takes, so that anything left to it comes too late."""
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


def dev(x):
    return torch.as_tensor(np.ascontiguousarray(x), device="cuda")


class BusyDefaultStream:
    """Copies on the default stream (0.3 ms each) and a side stream as the current one."""

    def __init__(self, copies=256):
        self.copies = copies

    def __enter__(self):
        self.a = torch.zeros(1 << 28, dtype=torch.float32, device="cuda")
        self.b = torch.empty_like(self.a)
        self.side = torch.cuda.stream(torch.cuda.Stream())
        torch.cuda.synchronize()
        for _ in range(self.copies):
            self.b.copy_(self.a)
        self.busy = torch.cuda.Event()
        self.busy.record()
        self.side.__enter__()
        return self

    def __exit__(self, *exc):
        self.side.__exit__(*exc)
        torch.cuda.synchronize()


@pytest.mark.parametrize("ng,P", [(300, 4096), (1100, 1024)])
def test_first_split_tiles(gw, ng, P):
    """The first launch whose last tiles meet in parts clears their counters (6 and 45 tiles: all of them
    in parts).  The same bits as on an idle GPU."""
    rng = np.random.default_rng(ng)
    M = dev(rng.standard_normal((P, ng)) + 1j * rng.standard_normal((P, ng)))
    ev, ec = dev(np.full(1, -2.0)), dev(np.full(P, 2.0))
    make = lambda: gw.Chi0((8, 8, 8), prec="ozaki", nslices=7)  # noqa: E731
    want = make().contract(ev, ec, M, [0.0])
    out = torch.empty_like(want)
    for copies in (256, 2048):  # again where a slow host let the copies end first
        h = make()
        torch.cuda.synchronize()
        with BusyDefaultStream(copies) as busy:
            h.contract(ev, ec, M, [0.0], out=out)
            h.sync()
            late = not busy.busy.query()
            got = out.clone()
            h.contract(ev, ec, M, [0.0], out=out)  # the counters are left at zero
            h.sync()
        assert torch.equal(got, want) and torch.equal(out, want)
        h.destroy()
        if late:
            break


def test_first_batch(gw):
    """A batch's job tables are uploaded when its graph is built: a handle made, loaded and run with the default
    stream busy."""
    import gwgen
    p = gwgen.make_problem((24, 24, 24), 4, 60, 600, 130, seed=3)
    t = {k: dev(getattr(p, k)) for k in ("gpsi", "cv", "ev", "cc", "ec", "gchi")}

    def load(**kw):
        h = gw.Chi0(p.grid, **kw)
        h.set_bands(0, 1, t["gpsi"], t["cc"], t["ec"])
        h.set_bands(0, 0, t["gpsi"], t["cv"], t["ev"])
        h.set_gsphere(0, t["gchi"])
        return h

    for kw in (dict(prec="fp64"), dict(prec="ozaki", nslices=7, mtxel="twofloat")):
        want = load(**kw).compute_batch([0], [0.0, 2.0])[0].clone()
        out = torch.empty_like(want).reshape(-1)
        torch.cuda.synchronize()
        with BusyDefaultStream():
            h = load(**kw)
            got = h.compute_batch([0], [0.0, 2.0], out=out)[0].clone()
            h.sync()
        assert float(torch.linalg.vector_norm(got - want) / torch.linalg.vector_norm(want)) < 1e-14
        h.destroy()
