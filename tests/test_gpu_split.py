"""The FP32 K build on tensor cores (operands split into two FP16 parts, csrc/kbuild_tc.cu), through
popcorn_kernel_matrix and popcorn_fit, at the edges of its tiles and of its dispatch rules, against
the FP64 product of the same points.

Bound per entry, from the arithmetic: an operand is represented to 2^-24 of itself (two of them), a
32-column chunk is truncated twice (2 ulps of partial sums, 2 * 2^-23 by Cauchy-Schwarz), and the
d / 32 chunks are added in FP32 (2^-24 a sum, the last two rounded away: twice that): together
(d / 32 + 8) 2^-24 |x| |y|.
"""
import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu

LINEAR = {"kind": "linear", "gamma": 1.0, "coef0": 0.0, "degree": 1, "sigma": 1.0}


@pytest.fixture(scope="module")
def pc():
    import paper_2501_05587_gb300 as m
    return m


def _bound(P, d):
    nrm = P.double().norm(dim=1)
    return (d / 32 + 8) * 2.0 ** -24 * nrm[:, None] * nrm[None, :] + 1e-37


@pytest.mark.parametrize("n,d", [(1, 500), (127, 478), (128, 512), (129, 513), (255, 640), (257, 479), (1025, 777),
                                 (1153, 600), (4100, 129)])
@pytest.mark.parametrize("pad", [0, 3], ids=["aligned", "strided"])
def test_split_matrix(pc, n, d, pad):
    g = torch.Generator(device="cuda").manual_seed(n * 7 + d)
    P = torch.randn(n, d + pad, generator=g, device="cuda")[:, :d] * 3.0 + 0.5
    if pad:
        P = torch.empty(n, d + pad, device="cuda")[:, :d].copy_(P)   # ldp = d + 3: rows not 16-byte aligned
    K, kd = pc.popcorn_kernel_matrix(P, LINEAR)
    E = P.double() @ P.double().T
    assert bool(((K.double() - E).abs() <= _bound(P, d)).all())
    assert torch.equal(K, K.T) and torch.equal(K.diagonal(), kd)
    Kf, kf = pc.popcorn_kernel_matrix(P, LINEAR, schedule="full")
    assert torch.equal(K, Kf) and torch.equal(kd, kf)


def test_split_exact_on_small_integers(pc):
    P = torch.randint(-3, 4, (300, 512), generator=torch.Generator().manual_seed(1)).float().cuda()
    K, _ = pc.popcorn_kernel_matrix(P, LINEAR)
    assert torch.equal(K.double(), P.double() @ P.double().T)


@pytest.mark.parametrize("what", ["wide_columns", "huge", "tiny", "sparse", "zero", "nonfinite"])
def test_split_refused_inputs(pc, what):
    """Points the split would not represent as FP32 does stay on CUDA cores: every entry within
    the FMA chain's (d + 2) 2^-24 sum_l |x_l y_l|, non-finite rows non-finite."""
    n, d = 200, 600
    P = torch.randn(n, d, generator=torch.Generator(device="cuda").manual_seed(5), device="cuda")
    if what == "wide_columns":
        P[:, 0] *= 1e7
    elif what == "huge":
        P *= 1e15
    elif what == "tiny":
        P *= 1e-15
    elif what == "sparse":
        P[torch.rand(n, d, device="cuda") < 0.9] = 0.0
    elif what == "zero":
        P.zero_()
    else:
        P[3, 5] = float("inf")
        P[7, 9] = float("nan")
    K, _ = pc.popcorn_kernel_matrix(P, LINEAR)
    ok = torch.isfinite(P).all(1)
    assert not torch.isfinite(K[~ok]).any() if what == "nonfinite" else bool(ok.all())
    X = P[ok].double()
    tol = (d + 2) * 2.0 ** -24 * (X.abs() @ X.abs().T) + 1e-37
    assert bool(((K[ok][:, ok].double() - X @ X.T).abs() <= tol).all())


@pytest.mark.parametrize("n", [1500, 2049])
@pytest.mark.parametrize("k_pass,sym_tile", [("full", 0), ("symmetric", 0), ("symmetric", 1)],
                         ids=["square", "packed", "packed_branch"])
def test_split_fit_layouts(pc, n, k_pass, sym_tile):
    """The split build's three stored layouts through one pass: E against the FP64 K."""
    d, k = 520, 5
    g = torch.Generator(device="cuda").manual_seed(n)
    P = torch.rand(n, d, generator=g, device="cuda")
    lab = torch.randint(0, k, (n,), generator=g, device="cuda", dtype=torch.int32)
    E = torch.empty(n, k, device="cuda")
    pc.popcorn_fit(P, k, LINEAR, lab, max_iter=1, check_convergence=False, k_pass=k_pass, sym_tile=sym_tile, E_out=E)
    o = oracle.step(oracle.kernel_matrix(P.cpu().numpy(), LINEAR), lab.cpu().numpy(), k)
    scale = float((P.double().norm(dim=1).max()) ** 2)
    assert np.abs(E.cpu().numpy() - o["E"]).max() <= 1e-5 * scale
