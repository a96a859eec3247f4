"""Scratch that idles in a Hamiltonian's pool between calls is there for the library's own
allocations when the device has no other memory left."""
import pytest

from edinputs import configs as C

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2210_03511_gb300 import build
    build.build()
    import paper_2210_03511_gb300 as pkg
    return pkg


def test_idle_scratch_is_given_back(P):
    import torch
    p = C.square32()
    b = P.Basis(p.sector)
    h = P.Hamiltonian(b, p.terms)
    size = h.store(P.ED_F32)
    x = torch.randn((8, h.dim), dtype=torch.float32, device="cuda")
    y = torch.empty_like(x)
    h.store_free()
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    before = torch.cuda.mem_get_info()[0]
    h.store(P.ED_F32)
    h.apply(x, y)  # 75 MB of scratch
    torch.cuda.synchronize()
    kept = before - torch.cuda.mem_get_info()[0] - size
    assert kept > 32 << 20
    # leave less than the plain recursion's three vectors below (28 MB), which what idles covers
    free = torch.cuda.mem_get_info()[0]
    fill = torch.empty((free - (24 << 20)) >> 21 << 21, dtype=torch.uint8, device="cuda")
    assert torch.cuda.mem_get_info()[0] < 3 * 4 * h.dim
    try:
        ev, rep = h.lanczos(n_eig=1, tol=1e-3, dtype=P.ED_F32, reorth=False, max_iter=20, raise_on_nonconv=False)
        assert rep.iters > 0
        h.apply(x, y)  # without scratch, or with what is there
        torch.cuda.synchronize()
    finally:
        del fill
        torch.cuda.empty_cache()
