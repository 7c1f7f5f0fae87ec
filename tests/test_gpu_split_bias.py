"""Mean signed error of the FP32 K build on tensor cores (csrc/kbuild_tc.cu: chunks of 32 columns added
with truncation, the last two additions of chunks rounded away from zero) against FP64.

A chunk is low by 3/4 ulp on average (two truncating additions that matter), the chunks' ulps add up
to about one of the sum (1 to 2 times 2^-24 of it), and two additions away from zero put back at most
half an ulp each: the mean lies within 1.5 ulp = 3 * 2^-24 |x| |y| times 1/2, so 1.5 * 2^-24.  Gaussian,
gamma / sigma^2 = 1 / (2 d), uniform points (|x|^2 about d / 3): the distance's 2 * 1.5 * 2^-24 d / 3 by
1 / (2 d) is half a 2^-24 of K, which is added to as much for K's own rounding."""
import math

import pytest
import torch

pytestmark = pytest.mark.gpu
U = 2.0 ** -24


def _points(kind, n, d):
    g = torch.Generator(device="cuda").manual_seed(d)
    f = torch.rand if kind == "uniform" else torch.randn
    return f(n, d, generator=g, device="cuda")


@pytest.mark.parametrize("kind", ["uniform", "normal"])
@pytest.mark.parametrize("d", [128, 160, 256, 784, 1500])
def test_mean_error_of_inner_products(kind, d):
    import paper_2501_05587_gb300 as pc
    n = 1500
    P = _points(kind, n, d)
    K, kd = pc.popcorn_kernel_matrix(P, pc.kernel_spec("linear"))
    X = P.double()
    E = X @ X.T
    nrm = X.norm(dim=1)
    e = (K.double() - E) / (nrm[:, None] * nrm[None, :]) * torch.sign(E)
    off = ~torch.eye(n, dtype=torch.bool, device="cuda")
    assert abs(float(e[off].mean())) <= 1.5 * U
    assert abs(float(e.diagonal().mean())) <= 1.5 * U


@pytest.mark.parametrize("d", [48, 64, 96])
def test_mean_error_of_the_gaussian_with_few_chunks(d):
    import paper_2501_05587_gb300 as pc
    n = 4000
    P = _points("uniform", n, d)
    K, _ = pc.popcorn_kernel_matrix(P, pc.kernel_spec("gaussian", gamma=1.0, sigma=math.sqrt(2 * d)))
    X = P.double()
    r = (X * X).sum(1)
    E = torch.exp(-(r[:, None] + r[None, :] - 2 * X @ X.T) / (2 * d))
    rel = ((K.double() - E) / E)[~torch.eye(n, dtype=torch.bool, device="cuda")]
    assert abs(float(rel.mean())) <= U
