"""The structure build beside an allocator with little room: it takes less scratch (more,
smaller chunks of rows) before it gives up, the structure is the same, and what does
not fit leaves nothing behind."""
import ctypes

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


class Arena:
    """cudaMalloc behind the allocator interface, with a limit on the bytes held at once."""

    def __init__(self, P):
        self.rt = ctypes.CDLL("libcudart.so.13")
        self.live = self.peak = 0
        self.limit = 1 << 62
        self.sizes = {}

        def alloc(n, stream, ctx):
            p = ctypes.c_void_p()
            if self.live + n > self.limit or self.rt.cudaMalloc(ctypes.byref(p), ctypes.c_size_t(max(n, 1))) != 0:
                return None
            self.sizes[p.value] = n
            self.live += n
            self.peak = max(self.peak, self.live)
            return p.value

        def free(p, n, stream, ctx):
            assert self.sizes.pop(p) == n
            self.live -= n
            self.rt.cudaFree(ctypes.c_void_p(p))

        self._fns = (P.ed.ALLOC_FN(alloc), P.ed.FREE_FN(free))
        self.struct = P.ed.ed_allocator(self._fns[0], self._fns[1], None)

    def basis(self, P, sector):
        b = P.Basis.__new__(P.Basis)
        b._sec, b._keep = P.ed._sector_struct(sector)
        b._arena = self
        b.n_sites = int(sector.n_sites)
        b.handle = ctypes.c_void_p()
        P.ed.check(P.ed.lib().ed_basis_build(ctypes.byref(b._sec), ctypes.byref(self.struct), None,
                                             ctypes.byref(b.handle)))
        d = ctypes.c_int64()
        P.ed.check(P.ed.lib().ed_basis_dim(b.handle, ctypes.byref(d)))
        b.dim = int(d.value)
        return b


CASES = {
    "one_row": lambda: C.chain(10, 1.0, 0.3, translations=True, n_up=0),
    "chain16": lambda: C.chain16(),
    "triangular24": lambda: C.triangular24(),
    "square26": lambda: C.square([[5, 1], [-1, 5]], 1.0, 0.5, irrep="A", point="rot"),
    "kagome24_Jchi": lambda: C.kagome([[4, 0], [0, 2]], 1.0, 0.2, 0.3, irrep="A", point="none"),
}


@pytest.mark.parametrize("segments", [1, 3])
@pytest.mark.parametrize("name", sorted(CASES))
def test_little_room(P, name, segments):
    import torch
    p = CASES[name]()
    arena = Arena(P)
    b = arena.basis(P, p.sector)
    h = P.Hamiltonian(b, p.terms)
    seg = 0 if segments == 1 else max(5, (b.dim // 3).bit_length())
    dt = torch.float64 if h.is_real else torch.complex128
    g = torch.Generator(device="cuda").manual_seed(1)
    x = torch.randn(b.dim, dtype=dt, device="cuda", generator=g)
    y, z = torch.empty_like(x), torch.full_like(x, float("nan"))
    held = arena.live
    size = h.store(seg_log2=seg)
    h.apply(x, y)
    torch.cuda.synchronize()
    h.store_free()
    assert arena.live == held
    # room for the structure, a sixteenth of it and 64 KB
    arena.limit = held + size + size // 16 + (1 << 16)
    h.store(seg_log2=seg)
    h.apply(x, z)
    torch.cuda.synchronize()
    assert torch.equal(y, z)
    h.store_free()
    # and half of what it needs
    arena.limit = held + size // 2
    with pytest.raises(P.EdError) as e:
        h.store(seg_log2=seg)
    assert e.value.name == "ED_ERR_NOMEM"
    assert arena.live == held and h.store_info()["bytes"] == 0
    arena.limit = 1 << 62
    h.close()
    b.close()
    assert arena.live == 0
