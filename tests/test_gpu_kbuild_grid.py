"""The FP32 K build on CUDA cores where its blocks take more than one tile (more than 512 tiles an SM:
csrc/kbuild_simt.cu; the first size has one a block), on points that the tensor-core build and the Gaussian's norm expansion refuse:
every row of a sample against FP64, with the multiply-adds' bound (d + 2) 2^-24 sum_l |p_il p_jl| and, for
the Gaussian from coordinate differences, (d + 8) 2^-24 (1 + d2 / (2 sigma^2)) of the value."""
import pytest
import torch

pytestmark = pytest.mark.gpu
U = 2.0 ** -24


@pytest.mark.parametrize("kind", ["linear", "gaussian"])
@pytest.mark.parametrize("n", [25217, 50561])
def test_blocks_with_several_tiles(n, kind):
    import paper_2501_05587_gb300 as pc
    d = 129 if kind == "linear" else 20
    g = torch.Generator(device="cuda").manual_seed(n)
    P = torch.randn(n, d, generator=g, device="cuda")
    if kind == "linear":
        P[:, 0] *= 1e7                      # a wide column
    else:
        P += 300.0                          # long rows, short distances
    kern = pc.kernel_spec(kind, gamma=1.0, coef0=0.0, degree=1, sigma=3.0)
    K, kd = pc.popcorn_kernel_matrix(P, kern)
    rows = torch.cat([torch.tensor([0, 127, 128, n - 1]), torch.randint(0, n, (200,))]).cuda()
    X = P.double()
    if kind == "linear":
        E = X[rows] @ X.T
        tol = (d + 2) * U * (X[rows].abs() @ X.T.abs())
    else:
        d2 = torch.cdist(X[rows], X, compute_mode="donot_use_mm_for_euclid_dist") ** 2
        E = torch.exp(-d2 / 9.0)
        tol = (d + 8) * U * (1 + d2 / 9.0) * E + 1e-37
    assert bool(((K[rows].double() - E).abs() <= tol).all())
    assert torch.equal(K[rows], K[:, rows].T) and torch.equal(K.diagonal(), kd)
