"""The FP32 K build on tensor cores (csrc/kbuild_tc.cu) and points whose rows differ in length: K_ij
of two short rows is as exact, relative to |p_i| |p_j|, as FP32 multiply-adds make it.

Bounds.  A row i of errors e_ij = (K_ij - p_i . p_j) / (|p_i| |p_j|) has a root mean square of at most
sqrt(d / 3) u, u = 2^-24: d roundings, independent, each at most u times a partial sum and that at most
|p_i| |p_j|, so u^2 / 3 of variance each.  (The multiply-adds reach about a thirtieth of it, two parts
in the range of FP16's normal numbers less.)  The largest is at most (d + 2) u
sum_l |p_il p_jl| / (|p_i| |p_j|), the multiply-adds' own bound, or that of the split build:
operands 2^-23 of themselves (4 u), a chunk of 32 columns truncated by at most 2 ulps (4 u),
d / 32 additions, the last two away from zero (2 u): (d / 32 + 10) u.
"""
import math

import pytest
import torch

pytestmark = pytest.mark.gpu
LINEAR = {"kind": "linear", "gamma": 1.0, "coef0": 0.0, "degree": 1, "sigma": 1.0}
U = 2.0 ** -24


def _check(P):
    import paper_2501_05587_gb300 as pc
    d = P.shape[1]
    K, kd = pc.popcorn_kernel_matrix(P, LINEAR)
    X = P.double()
    nrm = X.norm(dim=1)
    nrm = torch.where(nrm > 0, nrm, torch.ones_like(nrm))
    N = nrm[:, None] * nrm[None, :]
    E = X @ X.T
    e = (K.double() - E) / N
    serial = (d + 2) * U * (X.abs() @ X.abs().T) / N
    assert bool((e.abs() <= torch.maximum(serial, torch.full_like(serial, (d / 32 + 10) * U))).all())
    row = e.pow(2).mean(dim=1).sqrt()
    assert float(row.max()) <= math.sqrt(d / 3) * U, (float(row.max() / U), int(row.argmax()))
    assert torch.equal(K, K.T) and torch.equal(K.diagonal(), kd)
    return K.double(), E


@pytest.mark.parametrize("n,d", [(300, 512), (1300, 500)])
@pytest.mark.parametrize("what,f", [("long", 1e3), ("long", 1e7), ("long", 1e8), ("long", 1e11), ("short", 1e-3),
                                    ("short", 1e-7), ("short", 1e-10), ("decades", 3), ("decades", 8),
                                    ("decades", 11)])
def test_rows_of_different_length(n, d, what, f):
    g = torch.Generator(device="cuda").manual_seed(n + d)
    P = torch.randn(n, d, generator=g, device="cuda")
    if what == "decades":
        P *= 10.0 ** (f * (torch.rand(n, 1, generator=g, device="cuda") - 0.5))
    else:
        P[n // 3] *= f
        P[n - 1] = 0.0                       # a zero row takes no part in the rule
    others = torch.arange(n, device="cuda") != n // 3
    _check(P)
    if what != "decades":
        # among the other rows: the long row is the only one that lifts the scale
        import paper_2501_05587_gb300 as pc
        K, _ = pc.popcorn_kernel_matrix(P, LINEAR)
        X = P.double()[others]
        nrm = X.norm(dim=1)
        nrm = torch.where(nrm > 0, nrm, torch.ones_like(nrm))
        e = (K[others][:, others].double() - X @ X.T) / (nrm[:, None] * nrm[None, :])
        assert float(e.pow(2).mean(dim=1).sqrt().max()) <= math.sqrt(d / 3) * U


@pytest.mark.parametrize("small", [1e-3, 1e-8])
def test_blocks_of_columns_large_in_other_rows(small):
    """Every row and every column has a large entry; K between the two blocks is of small products
    only and keeps the multiply-adds' accuracy relative to sum_l |p_il p_jl|."""
    n, d = 400, 512
    g = torch.Generator(device="cuda").manual_seed(2)
    P = torch.rand(n, d, generator=g, device="cuda") + 0.5
    P[: n // 2, : d // 2] *= small
    P[n // 2:, d // 2:] *= small
    K, E = _check(P)
    A, B = slice(0, n // 2), slice(n // 2, n)
    rel = ((K[A, B] - E[A, B]) / E[A, B]).abs()
    assert float(rel.max()) <= (d + 2) * U
    assert float(rel.pow(2).mean().sqrt()) <= math.sqrt(d / 3) * U
