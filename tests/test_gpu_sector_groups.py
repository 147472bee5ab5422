"""Sector product with groups on both sides of the table's layouts (at most 16
elements, where an entry also marks the orbits of full size, and more), with
short orbits, against the full-basis oracle: projecting H psi equals the sector
product of the projected psi. GPU only."""
import numpy as np
import pytest

from ftk_inputs import characters, named, random_state, translations
from ftk_inputs.lattice import A1, A2, D_Z
from oracle import sparse

pytestmark = pytest.mark.gpu


def _inversion(cl):
    """The site permutation R -> d_z - R, which keeps the bond types."""
    cells = np.linalg.inv(np.stack([A1, A2])) @ np.linalg.inv(cl.supercell.astype(float))
    perm = []
    for l in range(cl.n_sites):
        f = (D_Z - cl.pos[l] - cl.pos) @ cells
        perm.append(int(np.flatnonzero(np.abs(f - np.round(f)).max(axis=1) < 1e-9)[0]))
    return np.array(perm)


@pytest.mark.parametrize("n,inverted,k", [(8, False, 1), (12, True, 0), (18, False, 2), (18, True, 0)])
def test_sector_product_commutes_with_projection(n, inverted, k):
    import paper_1802_02854_gb300 as ftk
    from paper_1802_02854_gb300 import build
    build.build()
    cl = named(n)
    perms, vecs = translations(cl)
    chi = characters(vecs, cl.momenta[k])
    if inverted:
        inv = _inversion(cl)
        perms = np.concatenate([perms, perms[:, inv]])
        chi = np.ones(len(perms), dtype=np.complex128)
    assert (len(perms) > 16) == (n == 18 and inverted)
    psi = random_state(n, 70 + n)
    ctx = ftk.Context(cl, -1.0, 0.1, "fp64")
    sec = ftk.Sector(ctx, perms, chi, n_slots=4)
    sec.project(psi, 0)
    sec.project(sparse.hv(cl, -1.0, 0.1, psi), 1)
    sec.hv(0, 2)
    want, got = sec.get(1), sec.get(2)
    sec.close()
    ctx.close()
    assert np.linalg.norm(got - want) <= 1e-12 * np.linalg.norm(want)
