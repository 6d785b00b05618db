"""Calls captured into a CUDA graph and replayed: a replay is a call on whatever its buffers hold then.

The launches of a captured call keep the arguments of the capture, so nothing in a workspace may
depend on a value that the host makes anew for every call.  Each test captures one call, replays the
graph several times with the inputs overwritten in place in between, and compares every replay to the
bit with a plain call on a workspace of its own.
"""
import pytest
import torch

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.fixture(scope="module")
def gk():
    from paper_2509_00388_b200 import binding
    binding.lib()
    return binding


def captured(call):
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        call()
    return graph


# a unit in one CTA, in CTAs of a cluster, and in CTAs that merge through the workspace
@pytest.mark.parametrize("rows,batch,hkv,dtype", [(544, 1, 8, torch.bfloat16), (544, 2, 8, torch.bfloat16), (4096, 1, 8, torch.bfloat16),
                                                  (32768, 1, 8, torch.bfloat16), (4096, 1, 3, torch.float32), (2080, 16, 8, torch.bfloat16)])
def test_captured_decode_attention(gk, rows, batch, hkv, dtype):
    gen = torch.Generator(device=DEV).manual_seed(rows)
    q = torch.empty((batch, 4 * hkv, 128), dtype=dtype, device=DEV)
    K, V = (torch.empty((batch, hkv, rows, 128), dtype=dtype, device=DEV) for _ in range(2))
    p = gk.decode_params(q, K, V)
    ws, plain_ws = gk.decode_workspace(p, DEV), gk.decode_workspace(p, DEV)
    out, want = (torch.empty(q.shape, dtype=torch.float32, device=DEV) for _ in range(2))
    for t in (q, K, V):
        t.normal_(generator=gen)
    gk.graphkv_decode_attention(p, q, K, V, want, plain_ws)
    graph = captured(lambda: gk.graphkv_decode_attention(p, q, K, V, out, ws))
    for _ in range(3):
        q.normal_(generator=gen)
        V.normal_(generator=gen)
        out.fill_(float("nan"))
        graph.replay()
        gk.graphkv_decode_attention(p, q, K, V, want, plain_ws)
        assert torch.equal(out, want)
    gk.graphkv_decode_attention(p, q, K, V, out, ws)          # a plain call on the replayed workspace
    assert torch.equal(out, want)


# every form of the score sweeps and of the rest of the path: one kernel whose CTAs wait for one another (one and
# two row tiles, both head dimensions, one and several units), two kernels (by switch, and more units than the GPU
# holds at once), short rows in one kernel, fp32, sources re-picked, budgets per layer, the streaming
# similarity sweep
@pytest.mark.parametrize("n,batch,hkv,over", [
    (16384, 1, 8, {}), (6013, 2, 2, {"window": 64}), (8191, 1, 8, {"head_dim": 64}), (5000, 1, 1, {"topk_nodes": 100}),
    (6013, 1, 2, {"two": True}), (4100, 40, 8, {}), (1003, 1, 8, {}), (700, 1, 2, {"dtype": torch.float32}),
    (9000, 1, 2, {"reselect": 1}), (6000, 3, 2, {"budgets": [300, 100, 7]}), (4500, 1, 4, {"rounds": 0}),
    (16384, 2, 8, {"topk_nodes": 150})])
def test_captured_compress(gk, monkeypatch, n, batch, hkv, over):
    if over.get("two"):
        monkeypatch.setenv("GRAPHKV_TWO_SCORE_KERNELS", "1")
    gen = torch.Generator(device=DEV).manual_seed(n)
    d, w, dtype = over.get("head_dim", 128), over.get("window", 32), over.get("dtype", torch.bfloat16)
    Q = torch.empty((batch, 4 * hkv, w, d), dtype=dtype, device=DEV)
    K, V = (torch.empty((batch, hkv, n + w, d), dtype=dtype, device=DEV) for _ in range(2))
    p = gk.make_params(K, Qw=Q, V=V, window=w, budget=300, pool_kernel=7, topk_nodes=over.get("topk_nodes", 16), neighbors=8,
                       rounds=over.get("rounds", 2), reselect=over.get("reselect", 0))
    ws, plain_ws = gk.alloc_workspace(p, DEV), gk.alloc_workspace(p, DEV)
    got, want = gk.alloc_outputs(p, K), gk.alloc_outputs(p, K)

    def call(out, scratch):
        if "budgets" in over:
            gk.graphkv_compress_layers(p, over["budgets"], Q, K, V, *out, scratch)
        else:
            gk.graphkv_compress(p, Q, K, V, *out, scratch)

    def draw():
        for t, scale in ((Q, 3.0), (K, 1.0), (V, 1.0)):
            t.normal_(generator=gen).mul_(scale)

    draw()
    call(want, plain_ws)
    graph = captured(lambda: call(got, ws))
    for _ in range(4):
        draw()
        for t in got + want:
            t.view(torch.uint8).fill_(0xFF)
        graph.replay()
        assert gk.graphkv_read_status(ws) == gk.OK
        call(want, plain_ws)
        for a, b in zip(got, want):
            assert torch.equal(a.view(torch.uint8), b.view(torch.uint8))


def test_captured_score_without_a_workspace(gk):
    gen = torch.Generator(device=DEV).manual_seed(3)
    Q = torch.empty((1, 32, 32, 128), dtype=torch.bfloat16, device=DEV).normal_(generator=gen)
    K = torch.empty((1, 8, 12032, 128), dtype=torch.bfloat16, device=DEV).normal_(generator=gen)
    p = gk.make_params(K, Qw=Q, window=32, pool_kernel=7)
    got, want = (torch.empty((1, 8, 12000), dtype=torch.float32, device=DEV) for _ in range(2))
    ws = gk.alloc_workspace(p, DEV)
    gk.graphkv_score_noalloc(p, Q, K, want)                    # (the first call on a device stays out of captures)
    graph = captured(lambda: gk.graphkv_score_noalloc(p, Q, K, got))
    for _ in range(4):
        K.normal_(generator=gen)
        graph.replay()
        assert gk.graphkv_read_status_noalloc(torch.device(DEV)) == gk.OK
        gk.graphkv_score(p, Q, K, want, ws)
        assert torch.equal(got, want)
