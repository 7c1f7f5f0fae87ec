"""The two streams of a batch with FP32 K: row by row where the batch has fewer blocks of 128 rows than
the block-row stream has CTAs, by block rows above.  The same instance alone and among many copies
gives the same labels, and objectives within the K stream's bar of 1e-6 of each other."""
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp32", "bf16"])
@pytest.mark.parametrize("n,k", [(701, 20), (130, 3), (1023, 64)])
def test_an_instance_alone_and_among_many(precision, n, k):
    import paper_2501_05587_gb300 as pc
    P = torch.from_numpy(synth.gaussian_blobs(n, 8, k, seed=n)).cuda()
    lab = torch.from_numpy(synth.init_labels(n, k, seed=k)).cuda()
    one = {"P": P, "init_labels": lab, "k": k, "kernel": pc.kernel_spec("polynomial")}
    kw = dict(max_iter=2, check_convergence=False, precision=precision)
    alone = pc.popcorn_fit_batched([dict(one)], **kw)
    copies = 900 // ((n + 127) // 128) + 1
    many = pc.popcorn_fit_batched([dict(one) for _ in range(copies)], **kw)
    # a launch a pass more (the label records): 2 passes and the objective
    assert many["info"]["kernel_launches"] - alone["info"]["kernel_launches"] >= 3
    for t in (0, copies // 2, copies - 1):
        assert torch.equal(many["labels"][t], alone["labels"][0])
        assert abs(many["objectives"][t] - alone["objectives"][0]) <= 1e-6 * abs(alone["objectives"][0])
