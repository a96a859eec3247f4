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


def test_one_pool(P):
    """A second Hamiltonian's call on a stream takes the scratch that idles there after the first
    one's (another stream may take memory of its own); freeing both gives all of it back."""
    import torch
    p = C.square32()
    b = P.Basis(p.sector)
    hs = [P.Hamiltonian(b, p.terms) for _ in range(2)]
    x = torch.randn((8, b.dim), dtype=torch.float32, device="cuda")
    y, z = torch.empty_like(x), torch.empty_like(x)
    for h in hs:
        h.store(P.ED_F32)
        h.apply(x[0], y[0])
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    hs[0].apply(x, y)
    torch.cuda.synchronize()
    taken = torch.cuda.mem_get_info()[0]
    assert taken < before
    hs[1].apply(x, z)
    torch.cuda.synchronize()
    assert torch.cuda.mem_get_info()[0] >= taken
    assert torch.equal(y, z)
    z.zero_()
    torch.cuda.synchronize()
    hs[1].apply(x, z, stream=torch.cuda.Stream())
    torch.cuda.synchronize()
    assert torch.equal(y, z)
    held = sum(h.store_info()["bytes"] for h in hs)
    for h in hs:
        h.close()
    assert torch.cuda.mem_get_info()[0] >= before + held // 2
