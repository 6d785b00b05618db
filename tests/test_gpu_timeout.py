"""The bounded device-side waits: a wait that runs out must end the kernel by itself, leave
GRAPHKV_ERR_TIMEOUT in the status word and leave the workspace usable.

The wait is made to run out on the host side only: the limit is shortened through
GRAPHKV_WAIT_CYCLES and a test hook makes the MMA issuer of the statistics sweep leave out one
arrival (the one that announces its first accumulator), so the epilogue's wait for it, the
issuer's wait for the buffer to come back and the producer's wait for a free stage all reach
their limit and drain.  A second hook makes every CTA of the kernel that runs both sweeps leave
out its announcement at the hand-over between the passes, so the wait for the unit's other chunks
runs out.  Nothing faults, traps or waits without a limit."""
import os

import pytest
import torch

from paper_2509_00388_b200 import workloads as wl

pytestmark = pytest.mark.gpu


# 3000 tokens: the one-kernel path of short rows (hook 1 without the two kernels), else the score kernels;
# 6000 tokens: always the score kernels
@pytest.mark.parametrize("hook,two_kernels,n", [("1", False, 3000), ("1", True, 3000), ("2", False, 3000), ("1", False, 6000), ("1", True, 6000),
                                                ("2", False, 6000)])
def test_a_wait_that_runs_out_is_reported_and_the_next_call_is_exact(hook, two_kernels, n):
    from paper_2509_00388_b200 import binding as gk
    gk.lib()
    dev = torch.device("cuda:0")
    cfg = wl.scaled(wl.LLAMA_32K, n_prefix=n, budget=64, n_q_heads=8, n_kv_heads=2, n_clusters=16)
    inp = wl.make_inputs(cfg)
    Qd, Kd = inp["Qw"].to(dev), inp["K"].to(dev)
    p = gk.make_params(Kd, Qw=Qd, window=cfg.window, pool_kernel=cfg.pool_kernel)
    ws = gk.alloc_workspace(p, dev)
    want = torch.empty((p.batch, p.n_kv_heads, cfg.n_prefix), dtype=torch.float32, device=dev)
    gk.graphkv_score(p, Qd, Kd, want, ws)
    assert gk.graphkv_read_status(ws) == gk.OK

    got = torch.empty_like(want)
    os.environ["GRAPHKV_WAIT_CYCLES"] = "2000000"           # about a millisecond
    os.environ["GRAPHKV_DEBUG_WITHHOLD_COMMIT"] = hook
    if two_kernels:
        os.environ["GRAPHKV_TWO_SCORE_KERNELS"] = "1"
    try:
        gk.graphkv_score(p, Qd, Kd, got, ws)
        status = gk.graphkv_read_status(ws)                 # synchronises: the kernels returned
    finally:
        os.environ.pop("GRAPHKV_WAIT_CYCLES", None)
        os.environ.pop("GRAPHKV_DEBUG_WITHHOLD_COMMIT", None)
        os.environ.pop("GRAPHKV_TWO_SCORE_KERNELS", None)
    assert status == gk.ERR_TIMEOUT
    assert "timed out" in gk.status_string(status)

    # the same workspace, a normal call: the status is clean again and the scores are bit-exact
    gk.graphkv_score(p, Qd, Kd, got, ws)
    assert gk.graphkv_read_status(ws) == gk.OK
    assert torch.equal(got, want)


# the streaming similarity sweep: the kernel that takes its bounds from a sample (3) and the sweep itself (4) leave out the
# arrival that announces their first product
@pytest.mark.parametrize("hook", ["3", "4"])
def test_a_wait_of_the_streaming_sweep_that_runs_out(hook):
    from paper_2509_00388_b200 import binding as gk
    gk.lib()
    dev = torch.device("cuda:0")
    gen = torch.Generator(device=dev).manual_seed(7)
    K, V = (torch.randn((1, 8, 8192 + 32, 128), generator=gen, device=dev).to(torch.bfloat16) for _ in range(2))
    Q = torch.randn((1, 32, 32, 128), generator=gen, device=dev).to(torch.bfloat16)
    p = gk.make_params(K, Qw=Q, V=V, window=32, budget=512, pool_kernel=7, topk_nodes=160, neighbors=32, rounds=2)
    ws = gk.alloc_workspace(p, dev)
    want, got = gk.alloc_outputs(p, K), gk.alloc_outputs(p, K)
    gk.graphkv_compress(p, Q, K, V, *want, ws)
    assert gk.graphkv_read_status(ws) == gk.OK
    os.environ["GRAPHKV_WAIT_CYCLES"] = "2000000"           # about a millisecond
    os.environ["GRAPHKV_DEBUG_WITHHOLD_COMMIT"] = hook
    try:
        gk.graphkv_compress(p, Q, K, V, *got, ws)
        status = gk.graphkv_read_status(ws)                 # synchronises: the kernels returned
    finally:
        os.environ.pop("GRAPHKV_WAIT_CYCLES", None)
        os.environ.pop("GRAPHKV_DEBUG_WITHHOLD_COMMIT", None)
    assert status == gk.ERR_TIMEOUT

    # the same workspace, a normal call: the status is clean again and the results are the same to the bit
    gk.graphkv_compress(p, Q, K, V, *got, ws)
    assert gk.graphkv_read_status(ws) == gk.OK
    for a, b in zip(got, want):
        assert torch.equal(a.view(torch.uint8), b.view(torch.uint8))
