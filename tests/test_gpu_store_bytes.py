"""The reported size of a structure of many chunks is what it holds of its allocator, and
the byte limit is exact."""
import pytest

from edinputs import configs as C
from test_gpu_store_scratch import Arena, P  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu

CASES = {
    "one_row": lambda: C.chain(10, 1.0, 0.3, translations=True, n_up=0),
    "chain16": lambda: C.chain16(),
    "triangular24": lambda: C.triangular24(),
    "square26": lambda: C.square([[5, 1], [-1, 5]], 1.0, 0.5, irrep="A", point="rot"),
    "kagome24_Jchi": lambda: C.kagome([[4, 0], [0, 2]], 1.0, 0.2, 0.3, irrep="A", point="none"),
}


@pytest.mark.parametrize("little_room", [False, True])
@pytest.mark.parametrize("name", sorted(CASES))
def test_bytes(P, name, little_room):  # noqa: F811
    arena = Arena(P)
    p = CASES[name]()
    b = arena.basis(P, p.sector)
    h = P.Hamiltonian(b, p.terms)
    held = arena.live
    size = h.store()
    assert arena.live - held == size == h.store_info()["bytes"]
    if little_room:  # many chunks
        arena.limit = held + size + size // 16 + (1 << 16)
        h.store_free()
        size = h.store()
        assert arena.live - held == size == h.store_info()["bytes"]
    assert h.store(max_bytes=size) == size
    with pytest.raises(P.EdError) as e:
        h.store(max_bytes=size - 1)
    assert e.value.name == "ED_ERR_NOMEM" and arena.live == held
    h.close()
    b.close()
    assert arena.live == 0
