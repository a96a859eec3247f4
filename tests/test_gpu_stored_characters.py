"""Real characters that differ from -1 and 1 by rounding (ed_basis_build takes |chi|^2 to
1e-9): real FP64 vectors take them as signs, matrix-free and from the stored structure,
one vector, several, several warps per slice and in a batch, so the results are the
same bits; the other kinds multiply by the character in both."""
import dataclasses

import numpy as np
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


@pytest.mark.parametrize("off", [0.0, 2.0 ** -52, 4e-10])
def test_characters_are_signs(P, off):
    import torch
    p = C.chain(14, 1.0, 0.3, translations=True, k=7)
    chi = np.array(p.sector.chi, dtype=complex)
    assert np.abs(np.abs(chi.real) - 1).max() < 1e-12 and (chi.real < 0).any()
    chi[1:] = np.sign(chi[1:].real) * (1 - off)
    s = dataclasses.replace(p.sector, chi=chi)
    h = P.Hamiltonian(P.Basis(s), p.terms)
    assert h.is_real
    for dt in (torch.float64, torch.float32):
        g = torch.Generator(device="cuda").manual_seed(2)
        x = torch.randn((3, h.dim), dtype=dt, device="cuda", generator=g)
        free, y, one = torch.empty_like(x), torch.empty_like(x), torch.empty_like(x)
        h.store_free()
        h.apply(x, free)
        h.store()
        h.apply(x, y)
        for v in range(3):
            h.apply(x[v], one[v])
        b = P.Batch([h])
        z = torch.empty(3 * h.dim, dtype=dt, device="cuda")
        b.apply(x.reshape(-1).contiguous(), z, nvec=3)
        torch.cuda.synchronize()
        assert torch.equal(y, free) and torch.equal(one, free) and torch.equal(z.reshape(3, -1), free)
        h.store_set_lanes(4)
        h.apply(x[0], one[0])
        torch.cuda.synchronize()
        # rows of at most 28 entries of at most 0.5 sqrt(14) times the largest element
        eps = np.finfo(np.float64 if dt == torch.float64 else np.float32).eps
        assert (one[0] - free[0]).abs().max().item() <= 64 * eps * 28 * 0.5 * 14 ** 0.5 * x.abs().max().item()
