"""Small sectors with long rows take the stored pass with eight entries in flight, up to
a number of blocks per SM and from a mean row length on: sectors on both sides of those
lines, one to eight vectors, against the pass with four warps per slice and the
matrix-free kernel, and a batch on both sides against its sectors.

Real vectors: the matrix-free kernel's bits.  Complex ones sum the same products in
another order: rows of at most 90 entries of size at most sqrt(|G|) <= sqrt(96), so
64 eps of the absolute row sum."""
import math

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


CASES = {
    # rows, mean entries per row: few (long rows), few slices but short rows, many slices
    "square16_A1": lambda: C.square([[4, 0], [0, 4]], 1.0, 0.5),
    "chain16": lambda: C.chain16(),
    "triangular24_Gamma": lambda: C.triangular24(),
    "square26_A": lambda: C.square([[5, 1], [-1, 5]], 1.0, 0.5, irrep="A", point="rot"),
    "kagome12_E1": lambda: C.kagome([[2, 0], [0, 2]], 1.0, 0.2, 0.3, irrep="E1"),
    "triangular24_k": lambda: C.triangular24_sectors()[7],
}


def _vectors(torch, shape, dt, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    return torch.randn(shape, dtype=dt, device="cuda", generator=g)


@pytest.mark.parametrize("nvec", [1, 2, 4, 8])
@pytest.mark.parametrize("name", sorted(CASES))
def test_both_sides(P, name, nvec):
    import torch
    p = CASES[name]()
    h = P.Hamiltonian(P.Basis(p.sector), p.terms)
    kinds = ([torch.float32, torch.float64] if h.is_real else []) + [torch.complex64, torch.complex128]
    for dt in kinds:
        x = _vectors(torch, (nvec, h.dim), dt, 2)
        free, y, cap = (torch.full_like(x, float("nan")) for _ in range(3))
        h.store_free()
        h.apply(x, free)
        h.store()
        h.apply(x, y)
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g):
            h.apply(x, cap)
        g.replay()
        torch.cuda.synchronize()
        assert torch.equal(y, cap)
        if not dt.is_complex:
            assert torch.equal(y, free)
        else:
            eps = np.finfo(np.float32 if dt == torch.complex64 else np.float64).eps
            scale = 64 * eps * 90 * math.sqrt(96.0) * x.abs().max().item()
            assert (y - free).abs().max().item() <= scale


@pytest.mark.parametrize("count", [1, 3, 40])
def test_batch_both_sides(P, count):
    """count copies of a sector of 897 slices: below and above the line."""
    import torch
    p = C.triangular24()
    h = P.Hamiltonian(P.Basis(p.sector), p.terms)
    h.store()
    b = P.Batch([h] * count)
    for dt in (torch.float32, torch.float64):
        for nvec in (1, 2):
            x = _vectors(torch, (count, nvec, h.dim), dt, 4)
            y = torch.full_like(x, float("nan"))
            b.apply(x.reshape(-1), y.reshape(-1), nvec=nvec)
            z = torch.empty_like(x)
            for k in range(count):
                for v in range(nvec):
                    h.apply(x[k, v], z[k, v])
            torch.cuda.synchronize()
            assert torch.equal(y, z)
