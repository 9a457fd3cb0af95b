"""CUDA-graph capture of the entry points a serving loop replays every step:
greedy verification, mixed-token sampling and token-tree verification captured
in one graph, replayed on new inputs, give the eager results bit for bit.
(verify at T > 0 with the fused distillation is covered in
test_gpu_distill_accepted.py.)"""
import pytest
import torch

from paper_2310_07177_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def osd():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    import paper_2310_07177_gb300 as pkg
    pkg.build_library()
    pkg.load_library()
    return pkg


def _inputs(seed):
    dev = torch.device("cuda")
    spec = W.VERIFY[2]
    v = W.verify_inputs(spec, seed=seed, device=dev)
    tree = W.tree_inputs(8, W.MEDUSA_TREE, 4096, torch.bfloat16, 1.0, seed=seed, device=dev, target_noise=0.8)
    g = torch.Generator(device=dev).manual_seed(seed)
    u = torch.rand(spec.B, generator=g, device=dev)
    return spec, v, tree, u


def test_graph_replay_matches_eager(osd):
    spec, v, tree, u = _inputs(W.seed_for(2))
    par = W.MEDUSA_TREE
    B, k, V = spec.B, spec.k, spec.V
    static = {"target": v["target"].clone(), "greedy": v["greedy_tokens"].clone(), "u": u.clone(),
              "z0": v["draft"][:, 0].contiguous(), "t0": v["target"][:, 0].contiguous(),
              "tz": tree["draft"].clone(), "tt": tree["target"].clone(), "ty": tree["tokens"].clone(),
              "tu": tree["uniforms"].clone()}
    ws = torch.empty(osd.osd_verify_workspace_size(B, k, V), dtype=torch.uint8, device="cuda")
    tws = torch.empty(osd.osd_verify_tree_workspace_size(8, len(par), 4096), dtype=torch.uint8, device="cuda")
    tok = torch.empty(B, dtype=torch.int32, device="cuda")

    def step():
        r0 = osd.osd_verify(None, static["target"], static["greedy"], None, 0.0, workspace=ws)
        osd.osd_mixed_sample(static["z0"], static["t0"], static["u"], 0.4, temperature=0.8, tokens=tok)
        rt = osd.osd_verify_tree(static["tz"], static["tt"], par, static["ty"], static["tu"], 1.0, workspace=tws)
        return r0, rt

    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(side):
        step()  # warm-up outside capture
    torch.cuda.current_stream().wait_stream(side)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        g0, gt = step()

    # new inputs into the captured buffers, then replay
    spec2, v2, tree2, u2 = _inputs(W.seed_for(2) + 7)
    static["target"].copy_(v2["target"])
    static["greedy"].copy_(v2["greedy_tokens"])
    static["u"].copy_(u2)
    static["z0"].copy_(v2["draft"][:, 0])
    static["t0"].copy_(v2["target"][:, 0])
    for a, b in (("tz", "draft"), ("tt", "target"), ("ty", "tokens"), ("tu", "uniforms")):
        static[a].copy_(tree2[b])
    graph.replay()
    torch.cuda.synchronize()

    e0 = osd.osd_verify(None, v2["target"], v2["greedy_tokens"], None, 0.0)
    etok, _ = osd.osd_mixed_sample(v2["draft"][:, 0].contiguous(), v2["target"][:, 0].contiguous(), u2, 0.4,
                                   temperature=0.8)
    et = osd.osd_verify_tree(tree2["draft"], tree2["target"], par, tree2["tokens"], tree2["uniforms"], 1.0)
    torch.cuda.synchronize()
    assert torch.equal(g0.accepted, e0.accepted) and torch.equal(g0.out_tokens, e0.out_tokens)
    assert torch.equal(g0.mismatch_mask, e0.mismatch_mask)
    assert torch.equal(tok, etok)
    for f in ("accepted", "path", "out_tokens", "last_node"):
        assert torch.equal(getattr(gt, f), getattr(et, f)), f


def _chain(osd, z, t, y, u, sync):
    """Calls back to back that read what the one before wrote (gradients as logits, accepted
    counts) and write over what it read, small enough that each starts as the last one ends."""
    g = [torch.zeros_like(z, dtype=torch.float32) for _ in range(2)]
    t32, w = t.float(), t.clone()
    rej = osd.DistillAcceptedResult(torch.zeros(3, device="cuda"), torch.zeros(3, z.shape[2], device="cuda"),
                                    torch.zeros(3, dtype=torch.int32, device="cuda"),
                                    torch.zeros(1, dtype=torch.int32, device="cuda"))
    out = []
    for i in range(12):
        kind = ("fkl", "rkl", "jsd", "tvd", "ce")[i % 5]
        osd.osd_distill(z, w[:, :-1], loss_kind=kind, dlogits=g[0])
        sync()
        osd.osd_distill(g[0], t32[:, :-1], loss_kind=kind, temperature=0.01, dlogits=g[1])  # reads g0 ...
        sync()
        osd.osd_distill(z, w[:, :-1], loss_kind="ce", dlogits=g[0])                            # ... and writes it
        sync()
        r = osd.osd_verify(z, w, y, u, 1.0, diagnostics=False)
        sync()
        osd.osd_distill_accepted(z, w, r.accepted, kind, out=rej)
        sync()
        tok, _ = osd.osd_mixed_sample(g[0][:, 0], g[1][:, 0], u[:, 0].contiguous(), 0.5, temperature=0.01)
        sync()
        r0 = osd.osd_verify(None, w, y, None, 0.0, diagnostics=False)
        sync()
        w.copy_(t).mul_(1.0 - 0.05 * i)  # other kernels write the logits between
        out += [g[0].clone(), g[1].clone(), r.out_tokens, rej.dlogits.clone(), rej.count.clone(), tok, r0.out_tokens]
    torch.cuda.synchronize()
    return out


def test_dependent_calls_back_to_back(osd):
    inp = W.verify_inputs(W.VerifySpec(3, 2, 2048, torch.bfloat16, 2.0, 1.0, 0.8, 1.0), seed=5)
    z, t, y, u = (inp[k].cuda() for k in ("draft", "target", "tokens", "uniforms"))
    a = _chain(osd, z, t, y, u, lambda: None)
    b = _chain(osd, z, t, y, u, torch.cuda.synchronize)
    assert len(a) == len(b)
    for i, (p, q) in enumerate(zip(a, b)):
        assert torch.equal(p, q), i


def test_capture_with_forked_streams_and_status(osd):
    """Captured calls that follow a memset (the status), an event of another stream, or a
    join of two streams: a graph's edges are then not between two kernels alone."""
    inp = W.verify_inputs(W.VerifySpec(3, 2, 4096, torch.bfloat16, 2.0, 1.0, 0.8, 1.0), seed=6)
    z, t, y, u = (inp[k].cuda() for k in ("draft", "target", "tokens", "uniforms"))
    st = torch.full((1,), 7, dtype=torch.int32, device="cuda")
    ga, gb = torch.zeros(3, 2, 4096, device="cuda"), torch.zeros(3, 2, 4096, device="cuda")
    other = torch.cuda.Stream()

    def step():
        main = torch.cuda.current_stream()
        other.wait_stream(main)
        with torch.cuda.stream(other):
            osd.osd_distill(z, t[:, :2], loss_kind="jsd", dlogits=gb)
            r0 = osd.osd_verify(None, t, y, None, 0.0)
        osd.osd_distill(z, t[:, :2], loss_kind="rkl", dlogits=ga, status=st)
        main.wait_stream(other)
        l, g = osd.osd_distill(gb, ga, loss_kind="fkl", temperature=0.01)
        return r0, osd.osd_verify(z, t, y, u, 1.0), l, g
    e0, e1, el, eg = step()
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        c0, c1, cl, cg = step()
    for x in (ga, gb):
        x.zero_()
    st.fill_(7)
    for _ in range(3):
        graph.replay()
    torch.cuda.synchronize()
    assert int(st) == 0 and torch.equal(el, cl) and torch.equal(eg, cg)
    assert torch.equal(e0.out_tokens, c0.out_tokens) and torch.equal(e1.out_tokens, c1.out_tokens)
