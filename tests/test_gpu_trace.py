"""trace K (csrc/iterate.cu: a cluster of blocks, four entries a load where diag K is 16-byte aligned)
through the objective of one assignment step on K = 0, whose J is the sum of diag K: whole numbers,
so the sum is exact in any order."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("off", [0, 1, 3])
@pytest.mark.parametrize("n", [2, 3, 5, 127, 2049, 4095, 16387])
def test_trace_of_diag(n, off):
    import paper_2501_05587_gb300 as pc
    K = torch.zeros(n, (n + 3) // 4 * 4, device="cuda")[:, :n]
    g = torch.Generator(device="cuda").manual_seed(n)
    kd = torch.randint(1, 1 << 20, (n + off,), generator=g, device="cuda").float()[off:]
    lab = torch.randint(0, 2, (n,), generator=g, device="cuda", dtype=torch.int32)
    for _ in range(3):
        assert pc.popcorn_assign_step(K, kd, lab, 2)["J"] == float(kd.double().sum())
