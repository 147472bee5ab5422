"""The one-launch product of small vectors against the tiled passes and the
oracle, at the sizes where its launch changes: below one block, at each block
size, at the last size with one amplitude per thread and beyond it, and on
both sides of the rule that picks it. GPU only."""
import numpy as np
import pytest

from ftk_inputs import named, random_state, random_vectors
from oracle import sparse

pytestmark = pytest.mark.gpu


def _product(ftk, cl, prec, vs, tile_bits):
    import torch
    B = vs.shape[0]
    ctx = ftk.Context(cl, -1.0, 0.1, prec, max_rhs=B, tile_bits=tile_bits)
    if prec == "df":
        hi = vs.astype(np.complex64)
        v = np.concatenate([hi, (vs - hi.astype(np.complex128)).astype(np.complex64)])
    else:
        v = vs.astype(np.complex128 if prec == "fp64" else np.complex64)
    out = ctx.hv(torch.from_numpy(v).cuda() if v.shape[0] > 1 else torch.from_numpy(v[0]).cuda())
    torch.cuda.synchronize()
    o = out.cpu().numpy().reshape(v.shape).astype(np.complex128)
    passes = ctx.plan_info()
    ctx.close()
    return (o[:B] + o[B:] if prec == "df" else o), passes


@pytest.mark.parametrize("prec,tol", [("fp64", 1e-12), ("df", 1e-12), ("fp32", 1e-6)])
@pytest.mark.parametrize("n,B", [(2, 1), (4, 8), (12, 2), (14, 1), (16, 4), (18, 1), (20, 1)])
def test_gather_matches_tiles_and_oracle(prec, tol, n, B):
    import paper_1802_02854_gb300 as ftk
    from paper_1802_02854_gb300 import build
    build.build()
    cl = named(n)
    vs = random_vectors(n, B, 400 + n)
    got, plan = _product(ftk, cl, prec, vs, 0)
    tiled, _ = _product(ftk, cl, prec, vs, 11)
    # one launch over the whole vector below the sizes at which the tiles win
    width = n + int(np.log2(B))
    assert plan == (1, n) if width <= (20 if prec == "df" else 18) else plan[0] > 1
    for j in range(B):
        ref = sparse.hv(cl, -1.0, 0.1, vs[j])
        assert np.linalg.norm(got[j] - ref) <= tol * np.linalg.norm(ref)
        assert np.linalg.norm(got[j] - tiled[j]) <= tol * np.linalg.norm(ref)


@pytest.mark.parametrize("n", [10, 20])
def test_gather_reductions_match_tiles(n):
    """The dots that the product's last block sums (one and several
    amplitudes per thread): mTPQ statistics against the tiled passes, to the
    tolerance of their parity with the oracle."""
    import paper_1802_02854_gb300 as ftk
    cl = named(n)
    psi = random_state(n, 5)
    res = []
    for tile_bits in (0, 9):
        ctx = ftk.Context(cl, -1.0, 0.1, "fp64", n_saved=1, tile_bits=tile_bits)
        ctx.set_state(psi, 0.5)
        res.append(ctx.tpq_step(6, 100))
        ctx.close()
    for a, b, tol in zip(res[0], res[1], (1e-12, 5e-11, 1e-10)):
        assert np.abs(a - b).max() < tol
