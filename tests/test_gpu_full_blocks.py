"""H.x of sectors whose rows fill a 16-site block that no element maps onto block 0
(the searches of test_host_full_blocks, on the device): matrix-free and stored against
the oracle's matrix, to 64 eps (|H| |x|)_i."""
import numpy as np
import pytest

import oracle
from edinputs import configs as C
from edinputs.vectors import state_vector

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


CASES = {
    "square32_none": lambda: C.square([[4, 4], [4, -4]], 1.0, 0.5, point="none", irrep="A", n_up=28, n_sublat=2,
                                      translations=False),
    "square32_rot": lambda: C.square([[4, 4], [4, -4]], 1.0, 0.5, point="rot", irrep="A", n_up=28, n_sublat=2,
                                     translations=False),
    "chain48": lambda: C.chain(48, 1.0, 0.3, n_up=46, n_sublat=3),
    "chain64": lambda: C.chain(64, 1.0, 0.3, n_up=63, n_sublat=4),
}


@pytest.mark.parametrize("name", sorted(CASES))
def test_full_blocks(P, name):
    import torch
    p = CASES[name]()
    b = P.Basis(p.sector)
    h = P.Hamiltonian(b, p.terms)
    reps, stab = oracle.basis(p.sector)
    assert b.dim == len(reps)
    m = p.sector.n_sites // p.sector.n_sublat
    assert (reps >> np.uint64(p.sector.n_sites - m) == (1 << m) - 1).any()  # block 0 full
    H = oracle.csr(p, reps, stab)
    X = state_vector(11, reps, complex_=False)
    x = torch.tensor(X, device="cuda")
    free, y = torch.empty_like(x), torch.empty_like(x)
    h.apply(x, free)
    h.store()
    h.apply(x, y)
    torch.cuda.synchronize()
    bound = 64 * np.finfo(np.float64).eps * (abs(H) @ np.abs(X)) + 1e-300
    assert np.all(np.abs(free.cpu().numpy() - H @ X) <= bound)
    assert torch.equal(y, free)
