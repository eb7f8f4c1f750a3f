"""How much device memory happens to be free has no part in the results: with most of it taken by another
allocation the same bits as before, as long as the call's buffers can be had."""
import gwgen
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

# the FP64 contraction's pieces (slices of 16384 pairs, 137 MB) on a grid that keeps the FFT kernel, and the
# route of two-float stage (a) (slices and last-axis output of 1.1 GB)
CASES = [(dict(prec="fp64", pair_chunk=16384), (18, 18, 18), 32, 512, 700, 300, 0.45e9),
         (dict(prec="ozaki", nslices=7, mtxel="twofloat"), (40, 40, 40), 12, 300, 3000, 900, 3e9)]


@pytest.mark.parametrize("kw,grid,nv,nc,ngpsi,ng,left", CASES)
def test_same_bits_with_little_memory_free(kw, grid, nv, nc, ngpsi, ng, left):
    if not torch.cuda.is_available():
        pytest.fail("GPU tests need a CUDA device")
    import paper_2509_23018_gb300 as gw
    p = gwgen.make_problem(grid, nv, nc, ngpsi, ng, seed=8)
    want = gw.from_problem(p, **kw).compute(0, [0.0])[0].clone()
    h = gw.from_problem(p, **kw)
    out = torch.empty_like(want).reshape(-1)
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    free, _ = torch.cuda.mem_get_info()
    taken = torch.empty(max(0, int(free - left)), dtype=torch.uint8, device="cuda")
    try:
        got = h.compute(0, [0.0], out=out)[0]
        h.sync()
        assert torch.equal(got, want)
    finally:
        del taken
        torch.cuda.empty_cache()
        h.destroy()
