"""Several vectors on stored structures: FP32 kinds go through a copy interleaved by
row, FP64 kinds (and captured calls, which get no scratch) vector by vector.  The
sums are those of the one-vector pass, so every y must be its bits."""
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
    "one_row": lambda: C.chain(10, 1.0, 0.3, translations=True, n_up=0),
    "remainder": lambda: C.chain(13, 1.0, 0.2, n_up=5),
    "complex": lambda: C.kagome([[2, 0], [0, 2]], 1.0, 0.2, 0.3, irrep="E1"),
}


def _vectors(torch, shape, dt, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    return torch.randn(shape, dtype=dt, device="cuda", generator=g)


@pytest.mark.parametrize("nvec", [2, 3, 4, 5, 6, 7, 8])
@pytest.mark.parametrize("name", sorted(CASES))
def test_vectors_together_and_alone(P, name, nvec):
    import torch
    p = CASES[name]()
    b = P.Basis(p.sector)
    h = P.Hamiltonian(b, p.terms)
    kinds = ([torch.float32, torch.float64] if h.is_real else []) + [torch.complex64, torch.complex128]
    many = max(5, int(math.ceil(math.log2(max(b.dim, 2) / 8))))
    for seg in (0, many):
        h.store(seg_log2=seg)
        for dt in kinds:
            x = _vectors(torch, (nvec, b.dim), dt, nvec)
            y, z, cap = (torch.empty_like(x) for _ in range(3))
            h.apply(x, y)
            for v in range(nvec):
                h.apply(x[v], z[v])
            torch.cuda.synchronize()
            assert torch.equal(y, z), (seg, dt)
            if nvec == 5:
                g = torch.cuda.CUDAGraph()
                with torch.cuda.graph(g):
                    h.apply(x, cap)
                g.replay()
                torch.cuda.synchronize()
                assert torch.equal(y, cap), (seg, dt)


def test_streams_share_a_hamiltonian(P):
    """Calls on two streams with different vectors, repeated: each has scratch of its own."""
    import torch
    p = CASES["remainder"]()
    b = P.Basis(p.sector)
    h = P.Hamiltonian(b, p.terms)
    h.store()
    xs = [_vectors(torch, (5, b.dim), torch.float32, 3 + k) for k in range(2)]
    want = []
    for x in xs:
        y = torch.empty_like(x)
        h.apply(x, y)
        want.append(y)
    st = [torch.cuda.Stream() for _ in range(2)]
    ys = [[torch.empty_like(xs[0]) for _ in range(20)] for _ in range(2)]
    torch.cuda.synchronize()
    for r in range(20):
        for k in range(2):
            h.apply(xs[k], ys[k][r], stream=st[k])
    torch.cuda.synchronize()
    for k in range(2):
        for y in ys[k]:
            assert torch.equal(y, want[k])


@pytest.mark.parametrize("nvec", [1, 3, 8])
def test_batch_vectors(P, nvec):
    """A batch's several vectors against each sector alone (complex: the batch takes the general
    coefficient tables, a sector of real coefficients the two-multiply-add ones, so up to rounding)."""
    import torch
    probs = C.all_sectors("square", [[4, 0], [0, 4]], 1.0, 0.5, n_sublat=2)[:6]
    hs = [P.Hamiltonian(P.Basis(q.sector), q.terms) for q in probs]
    for h in hs:
        h.store()
    batch = P.Batch(hs)
    off = batch.row_off
    for dt, eps in ((torch.complex64, np.finfo(np.float32).eps), (torch.complex128, np.finfo(np.float64).eps)):
        x = _vectors(torch, (batch.total * nvec,), dt, 9)
        y = torch.empty_like(x)
        batch.apply(x, y, nvec=nvec)
        for s, h in enumerate(hs):
            xs = x[nvec * int(off[s]):nvec * int(off[s + 1])].reshape(nvec, -1).contiguous()
            z = torch.empty_like(xs)
            h.apply(xs, z)
            torch.cuda.synchronize()
            ys = y[nvec * int(off[s]):nvec * int(off[s + 1])].reshape(nvec, -1)
            # rows of at most 64 elements of size at most sqrt(128): 64 eps of the absolute row sum
            scale = 64 * eps * 64 * math.sqrt(128.0) * xs.abs().max().item()
            assert (ys - z).abs().max().item() <= scale
