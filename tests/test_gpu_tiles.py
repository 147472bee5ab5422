"""Tiled products at the edges of their layouts against the oracle: the smallest
tile that fits a warp and the next smaller one (which runs as gather passes),
tiles of every size up to the largest, several columns, every coupling sign, and
FP64 vectors on both sides of the rule that picks the fixed-point pass (wide
ranges, zeros, tiny and huge scales, infinities). GPU only."""
import numpy as np
import pytest

from ftk_inputs import named, random_vectors
from oracle import sparse

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ftk():
    from paper_1802_02854_gb300 import build
    build.build()
    import paper_1802_02854_gb300 as m
    return m


def _product(ftk, cl, prec, vs, tile_bits, K=-1.0, J=0.1):
    import torch
    B = vs.shape[0]
    ctx = ftk.Context(cl, K, J, prec, max_rhs=B, tile_bits=tile_bits)
    if prec == "df":
        hi = vs.astype(np.complex64)
        v = np.concatenate([hi, (vs - hi.astype(np.complex128)).astype(np.complex64)])
    else:
        v = vs.astype(np.complex128 if prec == "fp64" else np.complex64)
    out = ctx.hv(torch.from_numpy(v).cuda() if v.shape[0] > 1 else torch.from_numpy(v[0]).cuda())
    torch.cuda.synchronize()
    o = out.cpu().numpy().reshape(v.shape).astype(np.complex128)
    ctx.close()
    return o[:B] + o[B:] if prec == "df" else o


@pytest.mark.parametrize("prec,tol", [("fp64", 1e-12), ("df", 1e-12), ("fp32", 1e-6)])
@pytest.mark.parametrize("n,tile_bits,B", [(12, 6, 1), (12, 7, 2), (12, 8, 1), (14, 10, 4), (14, 13, 1), (16, 12, 8)])
def test_tile_sizes(ftk, prec, tol, n, tile_bits, B):
    cl = named(n)
    vs = random_vectors(n, B, 900 + n + tile_bits)
    got = _product(ftk, cl, prec, vs, tile_bits)
    for j in range(B):
        ref = sparse.hv(cl, -1.0, 0.1, vs[j])
        assert np.linalg.norm(got[j] - ref) <= tol * np.linalg.norm(ref)


@pytest.mark.parametrize("K,J", [(-1.0, 0.0), (0.0, 1.0), (0.37, -0.23), (1e-3, 250.0), (0.0, 0.0)])
def test_fixed_point_couplings(ftk, K, J):
    cl = named(14)
    vs = random_vectors(14, 1, 77)
    got = _product(ftk, cl, "fp64", vs, 12, K, J)[0]
    ref = sparse.hv(cl, K, J, vs[0])
    assert np.linalg.norm(got - ref) <= 1e-12 * np.linalg.norm(ref)


@pytest.mark.parametrize("kind", ["gauss", "tiny", "huge", "wide", "one", "zero", "half"])
def test_fixed_point_ranges(ftk, kind):
    """Gaussian vectors and scaled ones (fixed point), vectors whose components
    span more than its digits (floating point), and ones with zeros: each
    component within 1e-13 of the sum of its terms' sizes, which the rounding of
    a few dozen terms in either arithmetic stays far below."""
    n = 14
    cl = named(n)
    rng = np.random.default_rng(8)
    v = random_vectors(n, 1, 31)[0]
    if kind == "tiny":
        v = v * 2.0 ** -960
    elif kind == "huge":
        v = v * 2.0 ** 1000
    elif kind == "wide":
        v = v * np.exp(-60 * rng.random(v.size))
    elif kind == "one":
        v = np.zeros_like(v)
        v[1234] = 1 - 2j
    elif kind == "zero":
        v = np.zeros_like(v)
    elif kind == "half":
        v[rng.random(v.size) < 0.5] = 0
    scale = 2.0 ** 960 if kind == "tiny" else 2.0 ** -1000 if kind == "huge" else 1.0
    got = _product(ftk, cl, "fp64", v[None], 12)[0] * scale
    ref = sparse.hv(cl, -1.0, 0.1, v * scale)
    x = np.arange(v.size)
    size = 3.0 * np.abs(v) * scale
    for i, j, _ in cl.bonds.tolist():
        size += 0.3 * np.abs(v[x ^ (1 << i) ^ (1 << j)]) * scale
    assert np.all(np.abs(got - ref) <= 1e-13 * size)


def test_non_finite_stays_local(ftk):
    """An infinite component reaches its partners only, as in floating point."""
    n = 14
    cl = named(n)
    v = random_vectors(n, 1, 5)[0]
    ref = sparse.hv(cl, -1.0, 0.1, v)
    v[77] = np.inf
    got = _product(ftk, cl, "fp64", v[None], 12)[0]
    touched = {77} | {77 ^ (1 << i) ^ (1 << j) for i, j, _ in cl.bonds.tolist()}
    rest = np.array([q for q in range(v.size) if q not in touched])
    assert not np.isfinite(got[77])
    assert np.linalg.norm(got[rest] - ref[rest]) <= 1e-12 * np.linalg.norm(ref[rest])
