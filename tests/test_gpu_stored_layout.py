"""The stored structure's layout (slices of 32 rows with interleaved entries) at
the edges of slices: sectors of one row, part of a slice, whole slices and a
remainder, rows without entries, one and about eight column segments.

The sum of a row runs over its entries in stored order on one lane, so with real
vectors and one segment y must be the matrix-free kernel's, bit for bit; every y
is held to the bound of test_gpu_parity against the oracle's matrix:
64 eps (|H| |x|)_i.
"""
import math

import numpy as np
import pytest

import oracle
from edinputs import configs as C
from edinputs.vectors import state_vector

pytestmark = pytest.mark.gpu

EPS64 = np.finfo(np.float64).eps


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
    "one_row": (1, lambda: C.chain(10, 1.0, 0.3, translations=True, n_up=0)),
    "part_of_a_slice": (6, lambda: C.chain(12, 1.0, 0.3, translations=True, n_up=2)),
    "one_over_a_slice": (33, lambda: C.chain(33, 1.0, 0.3, n_up=1)),
    "whole_slices": (64, lambda: C.chain(64, 1.0, 0.3, n_up=1)),
    "remainder": (1287, lambda: C.chain(13, 1.0, 0.2, n_up=5)),
    "long_rows": (12870, lambda: C.square([[4, 0], [0, 4]], 1.0, 0.5, point="none", irrep="A", translations=False)),
    "complex": (None, lambda: C.kagome([[2, 0], [0, 2]], 1.0, 0.2, 0.3, irrep="E1")),
}


@pytest.mark.parametrize("segments", [1, 8])
@pytest.mark.parametrize("name", sorted(CASES))
def test_slice_edges(P, name, segments):
    import torch
    dim, make = CASES[name]
    p = make()
    b = P.Basis(p.sector)
    assert dim is None or b.dim == dim
    h = P.Hamiltonian(b, p.terms)
    cplx = not h.is_real
    reps, stab = oracle.basis(p.sector)
    H = oracle.csr(p, reps, stab)
    seg = 0 if segments == 1 else max(5, int(math.ceil(math.log2(max(b.dim, 2) / segments))))
    X = np.stack([state_vector(31 + v, reps, complex_=cplx) for v in range(3)])
    x = torch.tensor(X, dtype=torch.complex128 if cplx else torch.float64, device="cuda")
    free, y3, y1 = torch.empty_like(x), torch.empty_like(x), torch.empty_like(x)
    h.apply(x, free)
    size = h.store(seg_log2=seg)
    h.apply(x, y3)
    for v in range(3):
        h.apply(x[v], y1[v])
    torch.cuda.synchronize()
    for y in (y3, y1):
        Y = y.cpu().numpy()
        for v in range(3):
            bound = 64 * EPS64 * (abs(H) @ np.abs(X[v])) + 1e-300
            assert np.all(np.abs(Y[v] - H @ X[v]) <= bound)
        if segments == 1 and not cplx:
            assert torch.equal(y, free)
    # the byte limit is exact
    assert h.store(seg_log2=seg, max_bytes=size) == size
    with pytest.raises(P.EdError) as e:
        h.store(seg_log2=seg, max_bytes=size - 1)
    assert e.value.name == "ED_ERR_NOMEM"
    assert h.store_info() == dict(entries=0, segments=0, codes=0, bytes=0)


@pytest.mark.parametrize("segments", [2, 3, 8])
@pytest.mark.parametrize("name", sorted(set(CASES) - {"complex"}))
def test_real_fp32_over_segments(P, name, segments):
    """One real FP32 vector over several segments, with more and with fewer than three
    entries per row and segment (two kernels): 64 eps (|H| |x|)_i of FP32."""
    import torch
    p = CASES[name][1]()
    b = P.Basis(p.sector)
    h = P.Hamiltonian(b, p.terms)
    reps, stab = oracle.basis(p.sector)
    H = oracle.csr(p, reps, stab)
    x32 = state_vector(37, reps, complex_=False).astype(np.float32)
    x = torch.tensor(x32, device="cuda")
    y = torch.full_like(x, float("nan"))
    h.store(P.ED_F32, seg_log2=max(5, int(math.ceil(math.log2(max(b.dim, 2) / segments)))))
    h.apply(x, y)
    torch.cuda.synchronize()
    X = x32.astype(np.float64)
    bound = 64 * np.finfo(np.float32).eps * (abs(H) @ np.abs(X)) + 1e-30
    assert np.all(np.abs(y.cpu().numpy().astype(np.float64) - H @ X) <= bound)
