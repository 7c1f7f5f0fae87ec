"""Bounded waits of the block-row K stream (csrc/reduce_tiles.cu, one fit and a batch) and of the
tensor-core K builds (csrc/kbuild_tc.cu), made to run out through the library's test hooks: one CTA's
first copies are left out and every wait of the launch gives up after the given time.  Nothing
faults or hangs: the call reports POPCORN_ERR_TIMEOUT, and the next one is the ordinary one."""
import time

import pytest
import torch

import synth

pytestmark = pytest.mark.gpu
TIMEOUT = 4   # POPCORN_ERR_TIMEOUT


@pytest.fixture(scope="module")
def pc():
    import paper_2501_05587_gb300 as m
    return m


def _times_out(pc, monkeypatch, hook, call):
    monkeypatch.setenv(hook, "200")
    t0 = time.perf_counter()
    with pytest.raises(pc.PopcornError) as e:
        call()
    monkeypatch.delenv(hook)
    assert e.value.status == TIMEOUT and "bounded wait" in str(e.value), str(e.value)
    assert time.perf_counter() - t0 < 60
    torch.cuda.synchronize()   # the context is intact


@pytest.mark.parametrize("check", [False, True], ids=["graph", "plain"])
def test_block_row_stream(pc, monkeypatch, check):
    n, k = 6145, 40
    P = torch.from_numpy(synth.gaussian_blobs(n, 6, 9, seed=1, box=3.0)).cuda()
    lab = torch.from_numpy(synth.init_labels(n, k, seed=2)).cuda()
    call = lambda: pc.popcorn_fit(P, k, pc.kernel_spec("gaussian", gamma=1.0, sigma=3.0), lab, max_iter=4,  # noqa: E731
                                  check_convergence=check, history=True)
    ref = call()
    _times_out(pc, monkeypatch, "POPCORN_TEST_SYM_STALL_MS", call)
    again = call()
    assert torch.equal(again["labels"], ref["labels"]) and again["objective"] == ref["objective"]
    assert again["info"]["J_history"] == ref["info"]["J_history"]


def test_batched_block_row_stream(pc, monkeypatch):
    # (1,000 blocks of 128 rows and more: batches of few are read row by row)
    wls = synth.batched_instances(160, seed=5, n_lo=600, n_hi=1500)
    inst = [{"P": torch.from_numpy(w.P).cuda(), "k": w.k, "kernel": w.kernel,
             "init_labels": torch.from_numpy(w.init_labels).cuda()} for w in wls]
    call = lambda: pc.popcorn_fit_batched(inst, max_iter=4, check_convergence=False)  # noqa: E731
    ref = call()
    _times_out(pc, monkeypatch, "POPCORN_TEST_SYM_STALL_MS", call)
    again = call()
    for t in range(len(inst)):
        assert torch.equal(again["labels"][t], ref["labels"][t])
        assert again["objectives"][t] == ref["objectives"][t]


@pytest.mark.parametrize("precision,n", [("fp32", 300), ("fp32", 4000), ("bf16", 300), ("bf16x3", 4000)])
def test_tensor_core_build(pc, monkeypatch, precision, n):
    """n = 300: one tile a CTA; n = 4,000: several."""
    P = torch.rand(n, 512, generator=torch.Generator(device="cuda").manual_seed(n), device="cuda")
    call = lambda: pc.popcorn_kernel_matrix(P, pc.kernel_spec("linear"), precision=precision)  # noqa: E731
    ref, kd = call()
    _times_out(pc, monkeypatch, "POPCORN_TEST_BUILD_STALL_MS", call)
    again, kd2 = call()
    assert torch.equal(again, ref) and torch.equal(kd2, kd)
