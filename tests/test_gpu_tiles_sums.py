"""Sums of the block-row K stream (csrc/reduce_tiles.cu) over clusters of any size and points in any
order: no further off than the row-major stream's, whose warp spreads a row over 32 lanes.

K = p p^T of points p = m / 4096, 205 <= m <= 4096, whose products are exact in FP32, so that E's
error is the sums' alone (and E's own rounding, 2^-24).  One large cluster: bar 3.2e-7 of E, 2.6e-7
for the sums (what 32 lanes' partial sums reach on 30,011 such entries, emulated in numpy, float32)
and 0.6e-7 for E; runs of 64 k columns one by one in FP32 reach 1.5e-6 at k = 100 and 4.5e-6 at 256.
Clusters of one size, in any order: the root mean square error is at most that of the 32 lanes'
sums of the same rows, emulated here addition by addition."""
import pytest
import torch

pytestmark = pytest.mark.gpu
LINEAR = {"kind": "linear", "gamma": 1.0, "coef0": 0.0, "degree": 1, "sigma": 1.0}


def _labels(order, n, k, g):
    if order == "sorted":
        return (torch.arange(n, device="cuda") * k // n).int()
    lab = torch.randint(0, k, (n,), generator=g, device="cuda", dtype=torch.int32)
    if order == "random":
        return lab
    one = torch.rand(n, generator=g, device="cuda") < 0.97
    if order == "dominant_last":
        one = torch.arange(n, device="cuda") > n // 30
    lab[one] = k - 2
    return lab


def _points(n, g):
    return torch.randint(205, 4097, (n, 1), generator=g, device="cuda").float() / 4096


def _exact(P, lab, k):
    """E and J in float64, from the sums of p."""
    p = P[:, 0].double()
    m = torch.bincount(lab.long(), minlength=k).double()
    s = torch.zeros(k, dtype=torch.float64, device="cuda").index_add_(0, lab.long(), p)
    mean = s / m.clamp(min=1)
    return p[:, None] * mean[None, :], float((p * p).sum() - (s * mean).sum())


def _lanes(V, lab, k):
    """The row-major stream's sums [rows, k], float32: lane l adds the float4 chunks l, l + 32, ... of a
    row one column after the other to its bins, then the 32 bins of a cluster are added in order."""
    n4 = V.shape[1] // 4
    lab = lab.long()
    acc = torch.zeros(V.shape[0], 32 * k, device="cuda")
    for q0 in range(0, n4, 32):
        lane = torch.arange(min(32, n4 - q0), device="cuda")
        for e in range(4):
            col = 4 * (q0 + lane) + e
            at = lane * k + lab[col]
            acc[:, at] += V[:, col]
    for j in range(4 * n4, V.shape[1]):
        acc[:, (j - 4 * n4) * k + lab[j]] += V[:, j]
    acc = acc.view(-1, 32, k)
    t = torch.zeros(V.shape[0], k, device="cuda")
    c = torch.arange(k, device="cuda")
    for s in range(32):
        t += acc[:, (s + c) % 32, c]
    return t


@pytest.mark.parametrize("order", ["random", "sorted", "dominant"])
@pytest.mark.parametrize("n,k", [(6145, 64), (20011, 33), (30011, 100), (30011, 256)])
def test_no_further_off_than_32_lanes(n, k, order):
    import paper_2501_05587_gb300 as pc
    g = torch.Generator(device="cuda").manual_seed(n * k)
    P, lab = _points(n, g), _labels(order, n, k, g)
    E = torch.empty(n, k, device="cuda")
    pc.popcorn_fit(P, k, LINEAR, lab, max_iter=1, check_convergence=False, E_out=E)
    rows = torch.randperm(n, generator=g, device="cuda")[:512]
    want = _exact(P, lab, k)[0][rows]
    m = torch.bincount(lab.long(), minlength=k).double()
    has = m > (1 if order != "dominant" else n // 2)
    old = (_lanes(P[rows] * P[:, 0][None, :], lab, k).double() / m.clamp(min=1)).float()
    rms = lambda X: float((X[:, has].double() / want[:, has] - 1).pow(2).mean().sqrt())  # noqa: E731
    assert rms(E[rows]) <= rms(old), (rms(E[rows]), rms(old))


@pytest.mark.parametrize("order", ["dominant", "dominant_last"])
@pytest.mark.parametrize("n,k", [(20011, 33), (20011, 100), (30011, 100), (30011, 256), (6145, 64)])
def test_sums_of_large_clusters(n, k, order):
    import paper_2501_05587_gb300 as pc
    g = torch.Generator(device="cuda").manual_seed(n + k)
    P, lab = _points(n, g), _labels(order, n, k, g)
    E = torch.empty(n, k, device="cuda")
    r = pc.popcorn_fit(P, k, LINEAR, lab, max_iter=1, check_convergence=False, E_out=E, history=True)
    want, J = _exact(P, lab, k)
    has = want[0] > 0
    rel = (E[:, has].double() / want[:, has] - 1).abs()
    assert float(rel.max()) <= 3.2e-7
    assert bool((E[:, ~has] == 0).all())
    assert abs(r["info"]["J_history"][0] - J) <= 1e-6 * J


@pytest.mark.parametrize("order", ["dominant", "dominant_last", "sorted"])
def test_batched_sums_of_large_clusters(order):
    import paper_2501_05587_gb300 as pc
    g = torch.Generator(device="cuda").manual_seed(3)
    inst, want = [], []
    for n, k in [(7990, 64), (129, 20), (4096, 64), (8000, 17), (513, 40), (12000, 64), (300, 4)]:
        P, lab = _points(n, g), _labels(order, n, k, g)
        inst.append({"P": P, "init_labels": lab, "k": k, "kernel": LINEAR})
        want.append(_exact(P, lab, k)[1])
    inst, want = inst * 4, want * 4      # (blocks for every CTA: batches of few are read row by row)
    r = pc.popcorn_fit_batched(inst, max_iter=0, check_convergence=False)
    for x, got, J in zip(inst, r["objectives"], want):
        assert abs(got - J) <= 1e-6 * J, (x["P"].shape, x["k"])
