"""The block-row K stream over the packed triangle (csrc/reduce_tiles.cu: FP32 K, more than 32 clusters,
n >= 6145), one pass against the oracle's step: E within the K stream's bar 1e-5 max_j |K_ij| and
labels equal except near-ties.  Sizes at the edges of its 128-row blocks and 32-column pieces,
and at the fewest and the most clusters."""
import numpy as np
import pytest
import torch

import oracle
import synth
from tests.parity import oracle_kernel_matrix

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pc():
    import paper_2501_05587_gb300 as m
    return m


@pytest.mark.parametrize("n,k", [(6145, 33), (6272, 64), (6273, 100), (6303, 256), (6177, 40), (6207, 255)])
def test_tiles_pass(pc, n, k):
    kern = {"kind": "gaussian", "gamma": 1.0, "coef0": 0.0, "degree": 1, "sigma": 3.0}
    P = synth.gaussian_blobs(n, 6, 9, seed=n, box=3.0)
    lab = synth.init_labels(n, k, seed=k)
    lab[lab == k // 2] = 0                      # an empty cluster
    lab[: n // 2] = lab[: n // 2] // 4          # runs of equal labels in four columns, and skewed sizes
    K = oracle_kernel_matrix(P, kern)
    o = oracle.step(K, lab, k)
    E = torch.empty(n, k, device="cuda")
    r = pc.popcorn_fit(torch.from_numpy(P).cuda(), k, kern, torch.from_numpy(lab).cuda(), max_iter=1,
                       check_convergence=False, k_pass="auto", E_out=E, history=True)
    Eg = E.cpu().numpy().astype(np.float64)
    assert np.all(np.abs(Eg - o["E"]).max(axis=1) <= 1e-5 * np.abs(K).max(axis=1))
    got = r["labels"].cpu().numpy()
    near = o["margin"] < 1e-6 * o["scale"]
    assert np.array_equal(got[~near], o["labels"][~near])
    assert abs(r["info"]["J_history"][0] - o["J"]) <= 1e-6 * abs(o["J"])
    again = pc.popcorn_fit(torch.from_numpy(P).cuda(), k, kern, torch.from_numpy(lab).cuda(), max_iter=1,
                           check_convergence=False, k_pass="auto")
    assert np.array_equal(again["labels"].cpu().numpy(), got) and again["objective"] == r["objective"]
