"""The native binding against the ctypes path behind it: the same results for
the same calls, and every call it does not take (or that fails) answered by the
checks of the Python code."""
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
    pkg._load_binding()
    return pkg


class _Nothing:
    """A binding that takes no call."""

    def __getattr__(self, name):
        return lambda *a: None


def _calls(osd):
    spec = W.VerifySpec(5, 3, 1003, torch.bfloat16, 2.0, 1.0, 0.8, 1.0)
    v = {k: x.cuda() for k, x in W.verify_inputs(spec, seed=9).items() if torch.is_tensor(x)}
    z, t, y, u = v["draft"], v["target"], v["tokens"], v["uniforms"]
    tree = W.tree_inputs(3, [-1, 0, 0, 1], 501, torch.float32, 1.0, seed=4)
    tr = {k: tree[k].cuda() for k in ("draft", "target", "tokens", "uniforms")}
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    mask = torch.tensor([[1, 0, 1]] * 5, dtype=torch.uint8, device="cuda")
    acc = torch.tensor([0, 3, 2, -1, 1], dtype=torch.int32, device="cuda")

    def keep():
        return torch.full((5, 3, 1003), 7.0, device="cuda")
    return {
        "verify": lambda: osd.osd_verify(z, t, y, u, 1.0),
        "verify int temperature, no diagnostics": lambda: osd.osd_verify(z, t, y, u, 1, diagnostics=False),
        "verify greedy": lambda: osd.osd_verify(None, t, y, None, 0.0),
        "verify out, stream": lambda: osd.osd_verify(z, t, y, u, 0.7, out=osd.osd_verify(z, t, y, u, 1.0), stream=side),
        "distill": lambda: osd.osd_distill(z, t[:, :3], None, "jsd", 0.3, temperature=0.7),
        "distill masked": lambda: osd.osd_distill(z, t[:, :3], mask, 1, dlogits=keep()),
        "distill rows": lambda: osd.osd_distill(z[:, 0], t[:, 0], loss_kind="ce"),
        "accepted": lambda: osd.osd_distill_accepted(z, t, acc, "fkl", out=osd.DistillAcceptedResult(
            torch.zeros(5, device="cuda"), torch.zeros(5, 1003, device="cuda"),
            torch.zeros(5, dtype=torch.int32, device="cuda"), torch.zeros(1, dtype=torch.int32, device="cuda"))),
        "mixed": lambda: osd.osd_mixed_sample(z[:, 0], t[:, 1], u[:, 0].contiguous(), 0.4),
        "mixed gap": lambda: osd.osd_mixed_sample(z[0, :1].expand(5, -1), t[:, 1], u[:, 0].contiguous(), 0.4,
                                                  cdf_gap=torch.zeros(5, device="cuda")),
        "tree": lambda: osd.osd_verify_tree(tr["draft"], tr["target"], [-1, 0, 0, 1], tr["tokens"], tr["uniforms"], 1.0),
        "empty": lambda: osd.osd_distill(z[:0, 0], t[:0, 0]),
    }


NAMES = ["verify", "verify int temperature, no diagnostics", "verify greedy", "verify out, stream", "distill",
         "distill masked", "distill rows", "accepted", "mixed", "mixed gap", "tree", "empty"]


@pytest.mark.parametrize("name", NAMES)
def test_native_equals_ctypes(osd, monkeypatch, name):
    call = _calls(osd)[name]
    taken = []
    real = osd._binding

    class Spy:
        def __getattr__(self, f):
            def go(*a):
                taken.append(getattr(real, f)(*a))
                return taken[-1]
            return go
    monkeypatch.setattr(osd, "_binding", Spy())
    a = call()
    assert taken and all(r is not None for r in taken)
    monkeypatch.setattr(osd, "_binding", _Nothing())
    b = call()
    torch.cuda.synchronize()
    assert type(a) is type(b) and len(a) == len(b)
    for x, y in zip(a, b):
        assert (x is None) == (y is None)
        if x is not None:
            assert x.dtype == y.dtype and x.shape == y.shape
            torch.testing.assert_close(x, y, rtol=0, atol=0, equal_nan=True)


def test_calls_it_does_not_take(osd):
    z, t = torch.randn(2, 3, 40, device="cuda"), torch.randn(2, 4, 40, device="cuda")
    y, u = torch.zeros(2, 3, dtype=torch.int32, device="cuda"), torch.rand(2, 4, device="cuda")
    with pytest.raises(ValueError, match="CUDA tensors only"):
        osd.osd_verify(z.cpu(), t, y, u, 1.0)
    with pytest.raises(ValueError, match="contiguous"):
        osd.osd_verify(z, t.transpose(0, 1).contiguous().transpose(0, 1), y, u, 1.0)
    with pytest.raises(ValueError, match="int32"):
        osd.osd_verify(z, t, y.long(), u, 1.0)
    with pytest.raises(TypeError, match="float32 or bfloat16"):
        osd.osd_verify(z.half(), t.half(), y, u, 1.0)
    with pytest.raises(osd.OsdError):
        osd.osd_verify(z, t, y, u, -1.0)
    with pytest.raises(KeyError):
        osd.osd_distill(z, t[:, :3], loss_kind="kl")
    with pytest.raises(osd.OsdError):
        osd.osd_distill(z, t[:, :3], temperature=0.0)
    with pytest.raises(ValueError, match="mask"):
        osd.osd_distill(z, t[:, :3], torch.ones(2, 3, device="cuda"))
    # a tensor subclass and a numpy temperature go the long way and give the same result
    class Sub(torch.Tensor):
        pass
    a = osd.osd_verify(z.as_subclass(Sub), t, y, u, __import__("numpy").float32(1.0))
    b = osd.osd_verify(z, t, y, u, 1.0)
    assert torch.equal(a.out_tokens, b.out_tokens) and torch.equal(a.accepted, b.accepted)
