"""Several FP32 vectors through the copy interleaved by row: every y is the one-vector
call's, bit for bit, for every lane layout of the copy (2, 4 and 8 padded vectors, rows
ending inside a slice), over one and several segments, for real, general complex and
axis-aligned coefficients (each real or purely imaginary), with the copy and without
(captured)."""
import math

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
    # 100,247 rows, 23 over a slice
    "square26_A": lambda: C.square([[5, 1], [-1, 5]], 1.0, 0.5, irrep="A", point="rot"),
    "triangular24_k": lambda: C.triangular24_sectors()[7],
    # axis-aligned: the characters of E1 are powers of i; chirality terms with real characters
    "square32_E1": lambda: C.square([[4, 4], [4, -4]], 1.0, 0.5, irrep="E1", point="rot", n_sublat=2, n_up=9,
                                    max_table_bytes=4 << 20),
    "kagome24_Jchi": lambda: C.kagome([[4, 0], [0, 2]], 1.0, 0.2, 0.3, irrep="A", point="none"),
}


@pytest.mark.parametrize("segments", [1, 3])
@pytest.mark.parametrize("name", sorted(CASES))
def test_copied(P, name, segments):
    import torch
    p = CASES[name]()
    h = P.Hamiltonian(P.Basis(p.sector), p.terms)
    h.store(P.ED_C64, seg_log2=0 if segments == 1 else int(math.ceil(math.log2(h.dim / segments))))
    assert h.store_info()["segments"] >= min(segments, 2)
    kinds = ([torch.float32] if h.is_real else []) + [torch.complex64]
    g = torch.Generator(device="cuda").manual_seed(6)
    for dt in kinds:
        x = torch.randn((8, h.dim), dtype=dt, device="cuda", generator=g)
        one = torch.empty_like(x)
        for v in range(8):
            h.apply(x[v], one[v])
        for nvec in range(2, 9):
            y = torch.full_like(x[:nvec], float("nan"))
            h.apply(x[:nvec], y)
            torch.cuda.synchronize()
            assert torch.equal(y, one[:nvec]), nvec
        cap, graph = torch.full_like(x, float("nan")), torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            h.apply(x, cap)
        graph.replay()
        torch.cuda.synchronize()
        assert torch.equal(cap, one)


@pytest.mark.parametrize("count", [1, 4, 12])
def test_batch_copied(P, count):
    """count copies of a sector of 897 slices, two to eight vectors."""
    import torch
    p = C.triangular24()
    h = P.Hamiltonian(P.Basis(p.sector), p.terms)
    h.store()
    b = P.Batch([h] * count)
    g = torch.Generator(device="cuda").manual_seed(7)
    for nvec in (2, 3, 5, 8):
        x = torch.randn((count, nvec, h.dim), dtype=torch.float32, device="cuda", generator=g)
        y = torch.full_like(x, float("nan"))
        b.apply(x.reshape(-1), y.reshape(-1), nvec=nvec)
        z = torch.empty_like(x)
        for k in range(count):
            for v in range(nvec):
                h.apply(x[k, v], z[k, v])
        torch.cuda.synchronize()
        assert torch.equal(y, z), nvec
