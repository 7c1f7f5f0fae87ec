"""The z reduction of batched mode (csrc/iterate.cu: small clusters of a block's 1,024 rows on a few lanes,
larger ones on a warp) through the objective of the initial labels: K = p p^T of points whose products
are exact in FP32, J against float64.  J is within the K stream's bar, 1e-6, at the edges of the rows a
block takes, of its lanes a cluster (k = 128, 129) and of what counts as large (256 rows)."""
import pytest
import torch

pytestmark = pytest.mark.gpu
LINEAR = {"kind": "linear", "gamma": 1.0, "coef0": 0.0, "degree": 1, "sigma": 1.0}


@pytest.mark.parametrize("skew", ["even", "one", "two"])
def test_objective_over_cluster_sizes(skew):
    import paper_2501_05587_gb300 as pc
    g = torch.Generator(device="cuda").manual_seed(11)
    inst, want = [], []
    for n, k in [(257, 4), (1024, 16), (1025, 17), (2049, 1), (2049, 2), (2048, 32), (3000, 33), (1500, 128),
                 (1500, 129), (2050, 256)]:
        P = torch.randint(205, 4097, (n, 1), generator=g, device="cuda").float() / 4096
        lab = torch.randint(0, k, (n,), generator=g, device="cuda", dtype=torch.int32)
        if skew != "even":
            big = torch.rand(n, generator=g, device="cuda") < 0.9
            lab[big] = k - 1
            if skew == "two":
                lab[big & (torch.arange(n, device="cuda") % 2 == 0)] = 0
        inst.append({"P": P, "init_labels": lab, "k": k, "kernel": LINEAR})
        p = P[:, 0].double()
        m = torch.bincount(lab.long(), minlength=k).double().clamp(min=1)
        s = torch.zeros(k, dtype=torch.float64, device="cuda").index_add_(0, lab.long(), p)
        want.append(float((p * p).sum() - (s * s / m).sum()))
    r = pc.popcorn_fit_batched(inst, max_iter=0, check_convergence=False)
    for x, got, J in zip(inst, r["objectives"], want):
        assert abs(got - J) <= 1e-6 * J, (x["P"].shape, x["k"])
