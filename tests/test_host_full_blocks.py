"""Representative search on the CPU (harness of test_host_representatives) where an
all-up 16-site block meets a block that no element maps onto block 0.

Rep_X of an unreachable block is the marker 0xFFFF, which 16-site blocks also have as
the true Rep of a full block: the block reaches MinRep with an empty Sym list.  Both
searches against the oracle's brute force, for groups that leave every block in
place and one that exchanges two of three."""
import dataclasses

import numpy as np
import pytest

import oracle
from edinputs import configs as C
from test_host_representatives import _call, harness  # noqa: F401  (fixture)


def _swap(p, m, X, Y):
    """p's sector with the exchange of blocks X and Y added to the identity."""
    g = np.arange(p.sector.n_sites, dtype=np.int32)
    x, y = np.arange(X * m, X * m + m), np.arange(Y * m, Y * m + m)
    g[x], g[y] = y, x
    ident = np.arange(p.sector.n_sites, dtype=np.int32)
    return dataclasses.replace(p.sector, perm=np.stack([ident, g]), spinflip=np.zeros(2, np.uint8),
                               chi=np.ones(2, complex))


def _square32(point, n_up):
    return C.square([[4, 4], [4, -4]], 1.0, 0.5, point=point, irrep="A", n_up=n_up, n_sublat=2,
                    translations=False).sector


SECTORS = {
    "square32_none": lambda: _square32("none", 16),
    "square32_none_28": lambda: _square32("none", 28),
    "square32_rot": lambda: _square32("rot", 16),
    "chain48_none": lambda: C.chain(48, 1.0, n_up=33, n_sublat=3).sector,
    "chain48_swap_1_2": lambda: _swap(C.chain(48, 1.0, n_up=20, n_sublat=3), 16, 1, 2),
    "chain48_swap_0_2": lambda: _swap(C.chain(48, 1.0, n_up=33, n_sublat=3), 16, 0, 2),
    "chain64_none": lambda: C.chain(64, 1.0, n_up=63, n_sublat=4).sector,
}


def _states(s, seed):
    """States with every choice of full blocks that n_up allows, the other spins at random,
    and their neighbours by one exchange."""
    rng = np.random.default_rng(seed)
    m = s.n_sites // s.n_sublat
    out = set()
    for full in range(1 << s.n_sublat):
        sites = [m * X + l for X in range(s.n_sublat) if full >> X & 1 for l in range(m)]
        rest = [i for i in range(s.n_sites) if i not in sites]
        if len(sites) > s.n_up:
            continue
        for _ in range(12):
            up = sites + [int(i) for i in rng.choice(rest, s.n_up - len(sites), replace=False)]
            out.add(sum(1 << (s.n_sites - 1 - i) for i in up))
            down = [i for i in range(s.n_sites) if i not in up]
            if down:
                up[int(rng.integers(len(up)))] = int(rng.choice(down))
                out.add(sum(1 << (s.n_sites - 1 - i) for i in up))
    return np.array(sorted(out), dtype=np.uint64)


@pytest.mark.parametrize("name", sorted(SECTORS))
def test_full_blocks(harness, name):  # noqa: F811
    s = SECTORS[name]()
    assert s.n_sites == 16 * s.n_sublat
    states = _states(s, 7)
    ref = [oracle.rep(s, int(x)) for x in states]
    for variant in (0, 1):
        rc, rep, g, ns, cp, own = _call(harness, s, states, variant)
        assert rc == 0, (rc, variant)
        for i, (r0, g0, n0, ssum) in enumerate(ref):
            assert int(rep[i]) == r0 and ns[i] == n0 and cp[i] == (abs(ssum) > 1e-9), (i, variant)
            assert oracle.apply(s, int(g[i]), int(states[i])) == r0
            assert own[i] == (r0 == int(states[i]))
