"""Rounding error of the products against that of the order in which they are
documented to sum, on Gaussian vectors and against extended precision. GPU only.

The expected error: rounding a sum of variance p adds c^2 p with c = 0.425 u, the
root mean square of half a unit in the last place, uniform within it, over the
logarithm of the magnitude (u = 2^-53, 2^-24). The variances of the partial sums
follow from the coefficients: an x or y bond adds the mean square of its two, a z
bond J/2 for one state in two. The bound leaves 12 % for FP64 (magnitudes are not
spread evenly), 20 % for FP32 (the coefficients are rounded too)."""
import numpy as np
import pytest

from ftk_inputs import named, random_vectors

pytestmark = pytest.mark.gpu

K = -1.0
U = {"fp64": 2.0 ** -53, "fp32": 2.0 ** -24}
SLACK = {"fp64": 1.12, "fp32": 1.20}


def _expected(cl, J, prec, chains):
    """chains: bond types summed one after the other, each chain from zero, the
    chains' sums added up, the diagonal last."""
    count = [int((cl.bonds[:, 2] == g).sum()) for g in range(3)]
    var = [(K * K / 16 + (K / 4 + J / 2) ** 2) / 2] * 2 + [(J / 2) ** 2 / 2]
    diag = (count[0] + count[1]) * (J / 4) ** 2 + count[2] * ((J + K) / 4) ** 2
    total = sum(c * v for c, v in zip(count, var)) + diag
    rounded = total + diag   # the last sum, and the diagonal's coefficient
    done = 0.0
    for chain in chains:
        part = 0.0
        for g in chain:
            for _ in range(count[g]):
                part += var[g]
                rounded += part * (0.5 if g == 2 else 1.0)   # parallel z bonds add nothing
        if done:
            rounded += part + done
        done += part
    return 0.425 * U[prec] * np.sqrt(rounded / total)


def _error(cl, J, prec, v, tile_bits):
    import torch
    import paper_1802_02854_gb300 as ftk
    from paper_1802_02854_gb300 import build
    build.build()
    v = v.astype(np.complex128 if prec == "fp64" else np.complex64)
    ctx = ftk.Context(cl, K, J, prec, tile_bits=tile_bits)
    got = ctx.hv(torch.from_numpy(v).cuda())
    torch.cuda.synchronize()
    got = got.cpu().numpy()
    ctx.close()
    x = np.arange(v.size, dtype=np.int64)
    num = den = 0.0
    for part, res in ((v.real, got.real), (v.imag, got.imag)):
        a = part.astype(np.longdouble)
        ref = np.zeros_like(a)
        for i, j, g in cl.bonds.tolist():
            anti = (((x >> i) ^ (x >> j)) & 1).astype(bool)
            ref += np.where(anti, (K / 4 + J / 2) if g < 2 else J / 2, (K / 4, -K / 4, 0.0)[g]) * a[x ^ (1 << i) ^ (1 << j)]
            ref += np.where(anti, -1.0, 1.0) * ((J + K) / 4 if g == 2 else J / 4) * a
        num += float(np.sum((res.astype(np.longdouble) - ref) ** 2))
        den += float(np.sum(ref ** 2))
    return np.sqrt(num / den)


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("n,J", [(12, 0.1), (16, -0.2)])
def test_one_launch_product(prec, n, J):
    """z bonds, x bonds on top of them, y bonds from zero."""
    cl = named(n)
    v = random_vectors(n, 1, 5)[0]
    assert _error(cl, J, prec, v, 0) <= SLACK[prec] * _expected(cl, J, prec, [(2, 0), (1,)])


@pytest.mark.parametrize("n,J", [(12, 0.1), (12, -0.2)])
def test_floating_point_pass(n, J):
    """FP64 in one tile, a vector with a neighbourhood of zeros (fixed point takes
    none): z, y and x bonds in one chain."""
    cl = named(n)
    v = random_vectors(n, 1, 5)[0]
    v[[77] + [77 ^ (1 << i) ^ (1 << j) for i, j, _ in cl.bonds.tolist()]] = 0
    assert _error(cl, J, "fp64", v, 12) <= SLACK["fp64"] * _expected(cl, J, "fp64", [(2, 1, 0)])
