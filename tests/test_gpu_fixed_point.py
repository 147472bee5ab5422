"""Componentwise accuracy of the tiled FP64 product, whichever arithmetic a vector
takes (64-bit fixed point or floating point), against sums in extended precision.
GPU only.

The bound: an output is a sum of one term per bond and of its diagonal, which a
chain of multiply-adds in 64-bit floating point rounds to within
(terms + 3) 2^-53 of the sum of its terms' sizes (one rounding per term, three
more for the diagonal's coefficient and the result). Every admitted vector has
to stay within it at every component."""
import numpy as np
import pytest

from ftk_inputs import named, omega_grid, random_vectors
from oracle import sparse

pytestmark = pytest.mark.gpu

N = 14
WIDE = np.longdouble


@pytest.fixture(scope="module")
def ftk():
    from paper_1802_02854_gb300 import build
    build.build()
    import paper_1802_02854_gb300 as m
    return m


def _product(ftk, cl, vs, tile_bits, K, J):
    import torch
    ctx = ftk.Context(cl, K, J, "fp64", max_rhs=vs.shape[0], tile_bits=tile_bits)
    out = ctx.hv(torch.from_numpy(vs if len(vs) > 1 else vs[0]).cuda())
    torch.cuda.synchronize()
    o = out.cpu().numpy().reshape(vs.shape)
    ctx.close()
    return o


def _terms(cl, K, J, a, sizes):
    """Sum of the terms of H a for a real vector in extended precision; sizes:
    of their absolute values."""
    x = np.arange(a.size, dtype=np.int64)
    a = a.astype(WIDE)
    out = np.zeros_like(a)
    fold = np.abs if sizes else (lambda t: t)
    for i, j, g in cl.bonds.tolist():
        anti = (((x >> i) ^ (x >> j)) & 1).astype(bool)
        c = np.where(anti, (K / 4 + J / 2) if g < 2 else J / 2, (K / 4, -K / 4, 0.0)[g]).astype(WIDE)
        d = np.where(anti, -1.0, 1.0) * ((J + K) / 4 if g == 2 else J / 4)
        out += fold(c * a[x ^ (1 << i) ^ (1 << j)]) + fold(d * a)
    return out


def _check(cl, K, J, v, got):
    bonds = len(cl.bonds)
    for part, res in ((v.real, got.real), (v.imag, got.imag)):
        err = np.abs(res.astype(WIDE) - _terms(cl, K, J, part, False))
        size = _terms(cl, K, J, part, True)
        assert np.all(err <= (bonds + 1 + 3) * WIDE(2.0) ** -53 * size)


def _ball(cl, v, centre):
    """A state and all its partners far below the rest."""
    q = [centre] + [centre ^ (1 << i) ^ (1 << j) for i, j, _ in cl.bonds.tolist()]
    v[q] *= 2.0 ** -60
    return v


def _vector(cl, kind):
    v = random_vectors(N, 1, 31)[0]
    x = np.arange(v.size)
    up = sum((x >> s) & 1 for s in range(N))
    if kind == "ball":
        v = _ball(cl, v, 4321)
    elif kind == "imag-ball":
        v = v.real + 1j * _ball(cl, v.imag.copy(), 77)
    elif kind in ("edge-30", "edge-70"):   # the states of |S^z| >= 5, closed under H at K = 0
        v = np.where(np.abs(2 * up - N) >= 10, v * 2.0 ** -float(kind[5:]), v)
    elif kind == "half":
        v[np.random.default_rng(8).random(v.size) < 0.5] = 0
    elif kind == "one":
        v = np.zeros_like(v)
        v[1234] = 1 - 2j
    elif kind == "spread":
        v = v * np.exp(-6 * np.random.default_rng(9).random(v.size))
    elif kind == "typical":   # a typical state after twenty steps
        for _ in range(20):
            v = 0.5 * v - sparse.hv(cl, -1.0, 0.1, v) / N
            v /= np.linalg.norm(v)
    elif kind == "real":
        v = v.real + 0j
    return v


@pytest.mark.parametrize("kind", ["gauss", "ball", "imag-ball", "edge-30", "edge-70", "half", "one", "spread", "typical",
                                  "real"])
@pytest.mark.parametrize("K,J", [(-1.0, 0.1), (0.0, 1.0), (0.4, -0.8)])
@pytest.mark.parametrize("tile_bits", [9, 12])
def test_every_component(ftk, kind, K, J, tile_bits):
    cl = named(N)
    v = _vector(cl, kind)
    _check(cl, K, J, v, _product(ftk, cl, v[None], tile_bits, K, J)[0])


@pytest.mark.parametrize("n", [7, 12, 15])
def test_sizes(ftk, n):
    """Vectors smaller and larger than the measuring launch's tiles, on an open
    chain of alternating bonds with one long bond."""
    class Chain:
        n_sites = n
        pos = np.stack([np.arange(n), np.zeros(n)], axis=1).astype(np.float64)
        bonds = np.array([[s, s + 1, s % 3] for s in range(n - 1)] + [[0, n - 1, 1]], dtype=np.int32)
    vs = random_vectors(n, 2, 17)
    got = _product(ftk, Chain, vs, 7, -1.0, 0.2)
    for v, g in zip(vs, got):
        _check(Chain, -1.0, 0.2, v, g)


def test_columns_choose_alone(ftk):
    """A block whose columns need different arithmetics equals the columns alone."""
    cl = named(N)
    vs = np.stack([_vector(cl, k) for k in ("gauss", "edge-70", "one", "real")])
    vs[2] = 0
    got = _product(ftk, cl, vs, 12, -1.0, 0.1)
    assert not got[2].any()
    for v, g in zip(vs, got):
        _check(cl, -1.0, 0.1, v, g)
        assert np.array_equal(g, _product(ftk, cl, v[None], 12, -1.0, 0.1)[0])


def test_measured_afresh(ftk):
    """A vector's product is the same bits whatever was multiplied before it: other
    vectors, wider and narrower blocks, a solve."""
    import torch
    cl = named(N)
    v = torch.from_numpy(_vector(cl, "gauss")).cuda()
    far = torch.from_numpy(np.stack([2.0 ** 60 * _vector(cl, k) for k in ("edge-70", "gauss", "one", "half")])).cuda()
    ctx = ftk.Context(cl, -1.0, 0.1, "fp64", max_rhs=4, tile_bits=12)
    first = ctx.hv(v).clone()
    block = torch.stack([v] * 4)
    for other in (far, block, far, far):
        ctx.hv(other)
        assert torch.equal(ctx.hv(v), first)
        assert torch.equal(ctx.hv(block), torch.stack([first] * 4))
    ctx.set_probe(0, v.cpu().numpy(), 0.0)
    ctx.shifted_cocg([0], omega_grid(-1.0, 1.0, 5), 0.5, tol=1e-6)
    ctx.hv(far[0].clone())
    assert torch.equal(ctx.hv(block), torch.stack([first] * 4))
    assert torch.equal(ctx.hv(v), first)
    ctx.close()


def test_captured_product(ftk):
    """A single product in a caller's graph, replayed on changing inputs."""
    import torch
    cl = named(N)
    ctx = ftk.Context(cl, -1.0, 0.1, "fp64", tile_bits=12)
    v = torch.zeros(1 << N, dtype=torch.complex128, device="cuda")
    out = torch.empty_like(v)
    graph = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(graph, stream=ctx.stream):
        ftk.ftk_hv(ctx.handle, v.data_ptr(), out.data_ptr(), 1)
    for kind, scale in (("gauss", 1.0), ("typical", 2.0 ** 30), ("edge-70", 1.0), ("gauss", 2.0 ** -40), ("gauss", 1.0)):
        x = scale * _vector(cl, kind)
        v.copy_(torch.from_numpy(x))
        graph.replay()
        torch.cuda.synchronize()
        _check(cl, -1.0, 0.1, x, out.cpu().numpy())
        direct = ctx.hv(v)
        torch.cuda.synchronize()
        _check(cl, -1.0, 0.1, x, direct.cpu().numpy())
    ctx.close()


def test_denormal_components(ftk):
    """Products of the smallest numbers are rounded, not dropped: within one
    quantum per term, and a half for each multiple that is formed."""
    cl = named(N)
    v = random_vectors(N, 1, 3)[0] * 2.0 ** -1050
    got = _product(ftk, cl, v[None], 12, -1.0, 0.1)[0]
    for part, res in ((v.real, got.real), (v.imag, got.imag)):
        err = np.abs(res.astype(WIDE) - _terms(cl, -1.0, 0.1, part, False))
        assert np.all(err <= 2 * len(cl.bonds) * WIDE(2.0) ** -1074)


@pytest.mark.parametrize("kind", ["gauss", "spread", "edge-30"])
def test_iteration_and_solve(ftk, kind):
    """States of both arithmetics through the epilogues of the iteration and the
    solve: the statistics against the oracle's products (each step's own
    rounding, 1e-12 over six steps), the Green's function against the same solve
    with the one-launch product, which is floating point throughout, to the
    solve's tolerance."""
    cl = named(N)
    psi = _vector(cl, kind)
    psi /= np.linalg.norm(psi)
    ctx = ftk.Context(cl, -1.0, 0.1, "fp64", n_saved=1, tile_bits=12)
    ctx.set_state(psi, 0.5)
    u, logq, h2 = ctx.tpq_step(6, 100)
    ctx.close()
    v, lq = psi, 0.0
    for k in range(6):
        w = sparse.hv(cl, -1.0, 0.1, v)
        assert abs(u[k] - np.vdot(v, w).real / N) < 1e-12
        assert abs(logq[k] - lq) < 1e-12
        v = 0.5 * v - w / N
        lq += np.log(np.linalg.norm(v))
        v /= np.linalg.norm(v)
    omega = omega_grid(-2.0, 2.0, 33)
    G = []
    for tile_bits in (0, 12):
        ctx = ftk.Context(cl, -1.0, 0.1, "fp64", max_rhs=2, tile_bits=tile_bits)
        ctx.set_probe(0, psi, 0.0)
        ctx.set_probe(1, psi.conj(), 0.3)
        g, _, _ = ctx.shifted_cocg([0, 1], omega, 0.2, tol=1e-11)
        G.append(g)
        g, _, _, *_ = ctx.shifted_cocg_ex([0, 1], omega + 0.2j, tol=1e-11, seed_switch=True)
        G.append(g)
        ctx.close()
    for g in G[1:]:
        assert np.abs(g - G[0]).max() <= 1e-9 * np.abs(G[0]).max()


@pytest.mark.parametrize("n,B", [(18, 2), (20, 1), (20, 4)])
@pytest.mark.parametrize("K,J", [(0.0, 1.0), (0.4, -0.2)])
def test_couplings_without_fixed_point(ftk, K, J, n, B):
    """An x or y coefficient of zero: one launch up to 2^22 amplitudes, through
    the block product, the iteration and the step on the caller's buffers; norm
    error within that of a chain over all terms."""
    import torch
    cl = named(n)
    vs = random_vectors(n, B, 12)
    ctx = ftk.Context(cl, K, J, "fp64", max_rhs=B, n_saved=1)
    assert ctx.plan_info() == (1, n)
    out = ctx.hv(torch.from_numpy(vs if B > 1 else vs[0]).cuda())
    torch.cuda.synchronize()
    got = out.cpu().numpy().reshape(vs.shape)
    ref = [sparse.hv(cl, K, J, v) for v in vs]
    bound = (len(cl.bonds) + 4) * 2.0 ** -53 * 2 * len(cl.bonds) * max(abs(K), abs(J))
    for v, g, r in zip(vs, got, ref):
        assert np.linalg.norm(g - r) <= bound * np.linalg.norm(v)
    psi = vs[0] / np.linalg.norm(vs[0])
    ell = 2.0
    ctx.set_state(psi, ell)
    u, _, h2 = ctx.tpq_step(2, 100)
    ctx.close()
    w = sparse.hv(cl, K, J, psi)
    assert abs(u[0] - np.vdot(psi, w).real / n) < 1e-12
    p = torch.from_numpy(psi).cuda()
    o = torch.empty_like(p)
    stats = ftk.ftk_tpq_step_noalloc(n, cl.bonds, K, J, ell, p.data_ptr(), o.data_ptr(),
                                     torch.cuda.current_stream().cuda_stream)
    assert abs(stats[0] - u[0]) < 1e-12 and abs(stats[1] - h2[0]) < 1e-9 * abs(h2[0])
    assert np.linalg.norm(o.cpu().numpy() - (ell * psi - w / n)) <= 1e-13
