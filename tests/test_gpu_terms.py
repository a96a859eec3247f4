"""Invariance of the bond set under the group, as ed_hamiltonian_create checks it: every
element must map every listed bond, zero couplings included, onto a listed bond of
the same coupling (to 1e-12 (1 + |J|))."""
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


@pytest.mark.parametrize("name,ok", [("ring", True), ("reversed pairs", True), ("split couplings", True),
                                     ("rounding", True), ("one coupling", False), ("one bond", False),
                                     ("zero bond", False), ("zero ring", True)])
def test_bond_set(P, name, ok):
    p = C.chain(8, 1.0, translations=True)
    bonds = [tuple(map(int, b)) for b in p.terms.bonds]
    J = [1.0] * len(bonds)
    far = sorted({tuple(sorted((int(g[bonds[0][0]]), int(g[bonds[0][1]])))) for g in np.asarray(p.sector.perm)})
    assert far == sorted(tuple(sorted(b)) for b in bonds)
    other = next((a, b) for a in range(8) for b in range(a + 1, 8) if (a, b) not in far)
    orbit = sorted({tuple(sorted((int(g[other[0]]), int(g[other[1]])))) for g in np.asarray(p.sector.perm)})
    if name == "reversed pairs":
        bonds = [(b, a) if i % 2 else (a, b) for i, (a, b) in enumerate(bonds)]
    elif name == "split couplings":
        bonds, J = bonds + bonds[:3], [1.0 if i > 2 else 0.5 for i in range(len(bonds))] + [0.5] * 3
    elif name == "rounding":
        J[0] += 1e-13
    elif name == "one coupling":
        J[0] += 1e-9
    elif name == "one bond":
        bonds, J = bonds[1:], J[1:]
    elif name == "zero bond":
        bonds, J = bonds + [other], J + [0.0]
    elif name == "zero ring":
        bonds, J = bonds + orbit, J + [0.0] * len(orbit)
    terms = dataclasses.replace(p.terms, bonds=np.asarray(bonds, np.int32), J=np.asarray(J, float))
    b = P.Basis(p.sector)
    if ok:
        P.Hamiltonian(b, terms).close()
    else:
        with pytest.raises(P.EdError) as e:
            P.Hamiltonian(b, terms)
        assert e.value.name == "ED_ERR_NOT_SYMMETRIC"
