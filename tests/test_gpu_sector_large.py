"""Sector product with more basis vectors than 27 bits can number (28 sites, the
trivial group: the sector is the full basis), on sampled rows against the rows
of the oracle. GPU only."""
import numpy as np
import pytest

from ftk_inputs import named
from oracle.rows import hv_rows

pytestmark = pytest.mark.gpu


def test_sector_index_above_27_bits():
    import paper_1802_02854_gb300 as ftk
    from paper_1802_02854_gb300 import build
    build.build()
    n = 28
    cl = named(n)
    rng = np.random.default_rng(28)
    v = rng.random(2 << n)
    v -= 0.5
    v = v.view(np.complex128)
    ctx = ftk.Context(cl, -1.0, 0.1, "fp32")
    sec = ftk.Sector(ctx, np.arange(n)[None], np.ones(1, dtype=np.complex128), n_slots=2)
    sec.set(0, v)
    sec.hv(0, 1)
    got = sec.get(1)
    sec.close()
    ctx.close()
    xs = np.unique(np.concatenate([rng.integers(0, 1 << n, 20000), [0, (1 << 27) - 1, 1 << 27, (1 << n) - 1]]))
    want = hv_rows(cl, -1.0, 0.1, lambda idx: v[idx], xs)
    assert np.linalg.norm(got[xs] - want) <= 1e-12 * np.linalg.norm(want)
