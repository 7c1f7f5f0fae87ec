"""The tensor-core K build's walk over its tiles (csrc/kbuild_tc.cu: bands of 8 row blocks, column pair by
column pair): every tile is built, for every number of 128-blocks up to four bands and a remainder
and both schedules.  Whole numbers up to 8 in magnitude are exact in BF16, and so are their inner
products in FP32: K is compared bit for bit."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["bf16", "bf16x3"])
@pytest.mark.parametrize("d,blocks", [(40, range(1, 36)), (82000, (1, 2, 3, 4, 5, 9))], ids=["short_rows", "long_rows"])
def test_every_tile_is_built(precision, d, blocks):
    import paper_2501_05587_gb300 as pc
    lin = pc.kernel_spec("linear")
    for T in blocks:
        n = 128 * T - (T % 3) * 5
        g = torch.Generator(device="cuda").manual_seed(T)
        P = torch.randint(-8, 9, (n, d), generator=g, device="cuda").float()
        if d > 1000:
            P[torch.rand(n, d, generator=g, device="cuda") < 0.9] = 0.0
        E = (P.double() @ P.double().T).float()
        for schedule in ("symmetric", "full"):
            K, kd = pc.popcorn_kernel_matrix(P, lin, precision=precision, schedule=schedule)
            assert torch.equal(K, E), (T, schedule)
            assert torch.equal(kd, E.diagonal())
