"""Several vectors without an interleaved copy (FP64 kinds; captured calls and small
sectors of the FP32 kinds): the one-vector passes of all vectors share one launch per
column segment, and every y is the one-vector call's, bit for bit."""
import ctypes
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


def _vectors(torch, shape, dt, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    return torch.randn(shape, dtype=dt, device="cuda", generator=g)


def _nodes(torch, call):
    """Nodes (kernels, memsets, copies) of one captured call."""
    rt = ctypes.CDLL("libcudart.so.13")
    s = torch.cuda.Stream()
    torch.cuda.synchronize()
    graph, n = ctypes.c_void_p(), ctypes.c_size_t()
    assert rt.cudaStreamBeginCapture(ctypes.c_void_p(s.cuda_stream), 2) == 0  # relaxed
    try:
        call(s)
    finally:
        assert rt.cudaStreamEndCapture(ctypes.c_void_p(s.cuda_stream), ctypes.byref(graph)) == 0
    assert rt.cudaGraphGetNodes(graph, None, ctypes.byref(n)) == 0
    assert rt.cudaGraphDestroy(graph) == 0
    return n.value


@pytest.mark.parametrize("kind", ["float64", "complex128", "complex64"])
def test_launches(P, kind):
    """As many launches for eight vectors as for one; a batch's too."""
    import torch
    dt = getattr(torch, kind)
    p = C.chain(13, 1.0, 0.2, n_up=5)
    h = P.Hamiltonian(P.Basis(p.sector), p.terms)
    for seg, want in ((0, 1), (9, 3)):
        h.store(seg_log2=seg)
        assert h.store_info()["segments"] == want
        for nvec in (1, 2, 8):
            x = _vectors(torch, (nvec, h.dim), dt, 3)
            y = torch.empty_like(x)
            h.apply(x, y)
            assert _nodes(torch, lambda s: h.apply(x, y, stream=s)) == want
    h.store()
    b = P.Batch([h, h])
    one = None
    for nvec in (1, 8):
        x = _vectors(torch, (b.total * nvec,), dt, 3)
        y = torch.empty_like(x)
        b.apply(x, y, nvec=nvec)
        n = _nodes(torch, lambda s: b.apply(x, y, nvec=nvec, stream=s))
        one = n if one is None else one
        assert n == one


@pytest.mark.parametrize("nvec", [2, 5, 8])
@pytest.mark.parametrize("segments", [2, 8])
def test_captured_real_fp32_over_segments(P, segments, nvec):
    """Captured calls take no copy; with two segments of 1,287 rows they take the pass for rows
    of three and more entries per segment, with eight the other one."""
    import torch
    p = C.chain(13, 1.0, 0.2, n_up=5)
    h = P.Hamiltonian(P.Basis(p.sector), p.terms)
    h.store(P.ED_F32, seg_log2=max(5, int(math.ceil(math.log2(h.dim / segments)))))
    x = _vectors(torch, (nvec, h.dim), torch.float32, 5)
    y, z = torch.empty_like(x), torch.full_like(x, float("nan"))
    for v in range(nvec):
        h.apply(x[v], y[v])
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        h.apply(x, z)
    g.replay()
    torch.cuda.synchronize()
    assert torch.equal(y, z)


@pytest.mark.parametrize("nvec", [2, 3, 8])
@pytest.mark.parametrize("kind", ["float32", "float64"])
def test_real_batch(P, kind, nvec):
    """Real sectors of unequal sizes in a batch against each alone."""
    import torch
    hs = []
    for p in (C.chain(12, 1.0, 0.3, translations=True, n_up=0, n_sublat=2), C.chain(12, 1.0, 0.3, n_up=5, n_sublat=2),
              C.chain(12, 1.0, 0.3, translations=True, k=6, n_up=4, n_sublat=2)):
        hs.append(P.Hamiltonian(P.Basis(p.sector), p.terms))
        hs[-1].store()
    b = P.Batch(hs)
    x = _vectors(torch, (b.total * nvec,), getattr(torch, kind), 8)
    y = torch.empty_like(x)
    b.apply(x, y, nvec=nvec)
    for s, h in enumerate(hs):
        part = slice(nvec * int(b.row_off[s]), nvec * int(b.row_off[s + 1]))
        xs, ys = x[part].reshape(nvec, -1), y[part].reshape(nvec, -1)
        z = torch.empty_like(xs)
        for v in range(nvec):
            h.apply(xs[v], z[v])
        torch.cuda.synchronize()
        assert torch.equal(ys, z)
