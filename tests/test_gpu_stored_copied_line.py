"""Several FP32 vectors on both sides of the line between the one-vector passes side by
side (all their blocks resident at once) and the copy interleaved by row: every y is the
one-vector call's, bit for bit, eager and captured; small sectors make no scratch."""
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


# 28,699 rows are 112 blocks a vector, 56,682 rows 222; the line lies at five blocks per SM
CASES = {
    "one_row": lambda: C.chain(10, 1.0, 0.3, translations=True, n_up=0),
    "triangular24_Gamma": lambda: C.triangular24(),
    "triangular24_k": lambda: C.triangular24_sectors()[7],
    "kagome18_Jchi": lambda: C.kagome([[3, 0], [0, 2]], 1.0, 0.2, 0.3, irrep="A", point="none"),
}


@pytest.mark.parametrize("name", sorted(CASES))
def test_line(P, name):
    import torch
    p = CASES[name]()
    h = P.Hamiltonian(P.Basis(p.sector), p.terms)
    h.store(P.ED_C64)
    g = torch.Generator(device="cuda").manual_seed(16)
    for dt in ([torch.float32] if h.is_real else []) + [torch.complex64]:
        x = torch.randn((8, h.dim), dtype=dt, device="cuda", generator=g)
        one = torch.empty_like(x)
        for v in range(8):
            h.apply(x[v], one[v])
        for nvec in range(2, 9):
            y, cap = (torch.full_like(x[:nvec], float("nan")) for _ in range(2))
            h.apply(x[:nvec], y)
            graph = torch.cuda.CUDAGraph()
            with torch.cuda.graph(graph):
                h.apply(x[:nvec], cap)
            graph.replay()
            torch.cuda.synchronize()
            assert torch.equal(y, one[:nvec]), nvec
            assert torch.equal(cap, one[:nvec]), nvec


def test_small_sectors_take_no_scratch(P):
    """Free device memory stays as it was over the first call with several vectors."""
    import torch
    p = C.triangular24()
    b = P.Basis(p.sector)
    h, warm = (P.Hamiltonian(b, p.terms) for _ in range(2))
    x = torch.randn((5, h.dim), dtype=torch.float32, device="cuda")
    y = torch.empty_like(x)
    for g in (h, warm):
        g.store()
        g.apply(x[0], y[0])
    warm.apply(x, y)  # the kernels of several vectors are loaded
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    h.apply(x, y)
    torch.cuda.synchronize()
    assert torch.cuda.mem_get_info()[0] >= before
