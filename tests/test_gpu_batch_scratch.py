"""Batched block Lanczos of FP32 vectors beside an allocator with just the room it needs
without the copy of its blocks interleaved by row: the copy may be made, but is given
back before the refinement's vectors are taken."""
import numpy as np
import pytest

from edinputs import configs as C
from test_gpu_store_scratch import Arena, P  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu


class Picky(Arena):
    """Refuses allocations of one size."""

    refused = None

    def __init__(self, P):
        super().__init__(P)
        inner = self._fns[0]

        def alloc(n, stream, ctx):
            return None if n == self.refused else inner(n, stream, ctx)

        self._outer = P.ed.ALLOC_FN(alloc)
        self.struct = P.ed.ed_allocator(self._outer, self._fns[1], None)


def test_refinement_has_room(P):  # noqa: F811
    p = C.triangular24()
    arena = Picky(P)
    b = arena.basis(P, p.sector)
    h = P.Hamiltonian(b, p.terms)
    h.store()
    batch = P.Batch([h] * 12)
    kw = dict(block=3, n_eig=1, tol=1e-7, max_iter=40, dtype=P.ED_F32, raise_on_nonconv=False, check_every=4)
    arena.refused = 4 * 4 * batch.total  # three vectors take a copy padded to four
    ev0, rep0 = batch.lanczos(**kw)
    arena.refused = None
    held = arena.live
    arena.limit = arena.peak
    ev1, rep1 = batch.lanczos(**kw)
    assert arena.live == held
    assert rep1.converged_sectors == rep0.converged_sectors == 12
    assert np.array_equal(ev0, ev1)
    batch.close()
    h.close()
    b.close()
    assert arena.live == 0
