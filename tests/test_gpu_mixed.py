"""GPU parity of osd_mixed_sample (Section 4.1, mixed sampling) against the
oracle: tokens bit-exact outside near-ties, for both dtypes, aligned and
unaligned rows, broadcast rows, ragged and large vocabularies, beta at both
ends and inside, two temperatures; the GPU's own draws pass a chi-square test
against the scipy mixture."""
import numpy as np
import pytest
import torch
from scipy.special import softmax
from scipy.stats import chisquare

import oracle
from paper_2310_07177_gb300 import workloads as W

pytestmark = pytest.mark.gpu
TIE = 1e-6


@pytest.fixture(scope="module")
def osd():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    import paper_2310_07177_gb300 as pkg
    pkg.build_library()
    pkg.load_library()
    return pkg


def _inputs(N, V, dtype, seed, spread=2.0):
    g = torch.Generator().manual_seed(seed)
    z = (torch.randn(N, V, generator=g) * spread).to(dtype)
    t = (z.float() * 0.8 + torch.randn(N, V, generator=g) * spread).to(dtype)
    u = torch.rand(N, generator=g)
    return z, t, u


def _check(osd, z, t, u, beta, tau):
    dev = torch.device("cuda")
    gap_g = torch.empty(z.shape[0], device=dev)
    tok, _ = osd.osd_mixed_sample(z.to(dev), t.to(dev), u.to(dev), beta, temperature=tau, cdf_gap=gap_g)
    torch.cuda.synchronize()
    ref_tok, ref_gap = oracle.mixed_sample(z, t, u, beta, float(np.float32(tau)))
    tok = tok.cpu().numpy()
    ok = ref_gap >= TIE
    bad = np.nonzero(ok & (tok != ref_tok))[0]
    assert bad.size == 0, f"tokens differ at {bad[:8]}: gpu {tok[bad[:8]]} oracle {ref_tok[bad[:8]]} gaps {ref_gap[bad[:8]]}"
    V = z.shape[-1]
    assert np.all((tok >= 0) & (tok < V))
    gg = gap_g.cpu().numpy()
    assert np.all(np.abs(gg[ok] - ref_gap[ok]) <= 2e-6), np.max(np.abs(gg[ok] - ref_gap[ok]))
    # near-ties: the GPU may take the neighbouring step, never a zero-weight entry
    ties = np.nonzero(~ok)[0]
    if ties.size:
        lq = oracle.log_softmax(z.reshape(-1, V)[ties], float(np.float32(tau)))
        lp = oracle.log_softmax(t.reshape(-1, V)[ties], float(np.float32(tau)))
        w = beta * np.exp(lp) + (1 - beta) * np.exp(lq)
        assert np.all(w[np.arange(ties.size), tok[ties]] > 0)
    return int(ties.size), int((tok[ties] != ref_tok[ties]).sum())


SHAPES = [  # (N, V, dtype)
    (3, 1, torch.float32),
    (5, 7, torch.bfloat16),
    (64, 100, torch.float32),
    (16, 4097, torch.bfloat16),
    (12, 32000, torch.bfloat16),
    (4, 33001, torch.bfloat16),
    (6, 32128, torch.float32),
    (3, 128256, torch.bfloat16),
    (2, 65539, torch.float32),
    (1, 33001, torch.bfloat16),    # one row: 16-byte loads with a ragged last chunk
    (1, 4099, torch.float32),
    (2, 1 << 21, torch.bfloat16),  # the largest vocabulary
    (2, 1 << 21, torch.float32),
]


@pytest.mark.parametrize("N,V,dtype", SHAPES)
@pytest.mark.parametrize("beta,tau", [(0.5, 1.0), (0.0, 0.7), (1.0, 1.3), (0.2, 0.7)])
def test_matches_oracle(osd, N, V, dtype, beta, tau):
    z, t, u = _inputs(N, V, dtype, seed=N * 7 + V)
    _check(osd, z, t, u, beta, tau)


def test_many_rows_at_full_vocabulary(osd):
    """2048 rows x 32000 bf16: every row outside a near-tie is exact.  With CDF
    steps about 1/V = 3e-5 wide, a few percent of rows fall within 1e-6 of an
    edge; they are counted and reported."""
    z, t, u = _inputs(2048, 32000, torch.bfloat16, seed=5)
    ties, differ = _check(osd, z, t, u, 0.5, 1.0)
    print(f"mixed sample 2048 x 32000: near-ties {ties}, of which differ {differ}")
    assert ties < 0.1 * 2048


def test_workload_full_size_sampled(osd):
    """The benchmark's launch: 65536 rows x 32000 bf16 (the distill buffer's rows), beta = 1/2,
    on the GPU at full size; 64 sampled rows are checked against the oracle."""
    spec = W.DISTILL[4]
    d = W.distill_inputs(spec, seed=W.seed_for(4), device="cuda")
    g = torch.Generator(device="cuda").manual_seed(2310071779)
    u = torch.rand(spec.N, generator=g, device="cuda")
    gap = torch.empty(spec.N, device="cuda")
    tok, _ = osd.osd_mixed_sample(d["draft"], d["target"], u, 0.5, cdf_gap=gap)
    torch.cuda.synchronize()
    sel = torch.randperm(spec.N, generator=torch.Generator().manual_seed(1))[:64]
    z, t = d["draft"][sel.cuda()].cpu(), d["target"][sel.cuda()].cpu()
    ref, ref_gap = oracle.mixed_sample(z, t, u[sel.cuda()].cpu(), 0.5)
    got = tok[sel.cuda()].cpu().numpy()
    ok = ref_gap >= TIE
    assert np.array_equal(got[ok], ref[ok]), np.nonzero(got[ok] != ref[ok])
    assert np.all(np.abs(gap[sel.cuda()].cpu().numpy()[ok] - ref_gap[ok]) <= 2e-6)
    assert bool(((tok >= 0) & (tok < spec.V)).all())


def test_strided_and_broadcast_rows(osd):
    dev = torch.device("cuda")
    g = torch.Generator().manual_seed(3)
    big_z = torch.randn(6, 3, 5000, generator=g).to(torch.bfloat16)
    big_t = torch.randn(6, 4, 5000, generator=g).to(torch.bfloat16)
    u = torch.rand(6, generator=g)
    z, t = big_z[:, 1], big_t[:, 2]  # row strides 3V and 4V
    tok, _ = osd.osd_mixed_sample(big_z.to(dev)[:, 1], big_t.to(dev)[:, 2], u.to(dev), 0.3)
    torch.cuda.synchronize()
    ref, gap = oracle.mixed_sample(z, t, u, 0.3)
    assert np.array_equal(tok.cpu().numpy()[gap >= TIE], ref[gap >= TIE])
    # padded rows: 16-byte aligned strides around a ragged vocabulary of 5003
    pz = torch.randn(6, 5008, generator=g).to(torch.bfloat16)
    pt = torch.randn(6, 5008, generator=g).to(torch.bfloat16)
    tok, _ = osd.osd_mixed_sample(pz.to(dev)[:, :5003], pt.to(dev)[:, :5003], u.to(dev), 0.6)
    torch.cuda.synchronize()
    ref, gap = oracle.mixed_sample(pz[:, :5003].contiguous(), pt[:, :5003].contiguous(), u, 0.6)
    assert np.array_equal(tok.cpu().numpy()[gap >= TIE], ref[gap >= TIE])
    # stride 0: one row repeated
    zr = z[:1].expand(6, -1)
    tr = t[:1].expand(6, -1)
    tok, _ = osd.osd_mixed_sample(zr.to(dev), tr.to(dev), u.to(dev), 0.3)
    torch.cuda.synchronize()
    ref, gap = oracle.mixed_sample(zr.contiguous(), tr.contiguous(), u, 0.3)
    assert np.array_equal(tok.cpu().numpy()[gap >= TIE], ref[gap >= TIE])


def test_neg_inf_entries_are_never_drawn(osd):
    N, V = 64, 3000
    z, t, u = _inputs(N, V, torch.float32, seed=9)
    z[:, ::3] = float("-inf")
    t[:, ::3] = float("-inf")
    u[:4] = 0.0
    _check(osd, z, t, u, 0.4, 1.0)
    tok, _ = osd.osd_mixed_sample(z.cuda(), t.cuda(), u.cuda(), 0.4)
    assert torch.all(tok % 3 != 0)


def test_gpu_draws_follow_the_mixture(osd):
    V, n, beta, tau = 8, 1_000_000, 0.35, 0.8
    g = torch.Generator().manual_seed(21)
    z1 = torch.randn(V, generator=g) * 1.5
    t1 = torch.randn(V, generator=g) * 1.5
    u = torch.rand(n, generator=g)
    dev = torch.device("cuda")
    tok, _ = osd.osd_mixed_sample(z1.to(dev).expand(n, V), t1.to(dev).expand(n, V), u.to(dev), beta,
                                  temperature=tau)
    counts = np.bincount(tok.cpu().numpy(), minlength=V)
    tau32 = float(np.float32(tau))
    mix = beta * softmax(t1.double().numpy() / tau32) + (1 - beta) * softmax(z1.double().numpy() / tau32)
    _, pval = chisquare(counts, mix * n)
    assert pval > 1e-4, (counts, mix * n)


def test_invalid_arguments_are_rejected(osd):
    dev = torch.device("cuda")
    z = torch.zeros(2, 16, device=dev)
    u = torch.zeros(2, device=dev)
    for beta, tau in ((1.5, 1.0), (-0.1, 1.0), (0.5, 0.0), (0.5, float("inf"))):
        with pytest.raises(osd.OsdError) as ei:
            osd.osd_mixed_sample(z, z, u, beta, temperature=tau)
        assert ei.value.status == osd.OSD_ERR_INVALID_ARG
    big = torch.zeros(1, (1 << 21) + 1, dtype=torch.bfloat16, device=dev)
    with pytest.raises(osd.OsdError) as ei:
        osd.osd_mixed_sample(big, big, u[:1], 0.5)
    assert ei.value.status == osd.OSD_ERR_UNSUPPORTED
    with pytest.raises(ValueError):
        osd.osd_mixed_sample(z, z, u.double(), 0.5)
    e = torch.zeros(0, 16, device=dev)
    tok, _ = osd.osd_mixed_sample(e, e, torch.zeros(0, device=dev), 0.5)
    assert tok.numel() == 0


# Rows off the 16-byte grid: both rows of a pair at the same phase (chunks cut there), or at
# different ones (chunks shifted into place): `shift` entries between the two.
@pytest.mark.parametrize("N,V,dtype,shift", [
    (40, 3, torch.bfloat16, 0), (40, 9, torch.bfloat16, 0), (9, 255, torch.float32, 0), (33, 4099, torch.bfloat16, 0),
    (9, 32001, torch.bfloat16, 0), (9, 32004, torch.bfloat16, 0), (5, 33003, torch.float32, 0),
    (40, 9, torch.bfloat16, 3), (9, 1023, torch.float32, 1), (9, 32001, torch.bfloat16, 5), (3, 128257, torch.bfloat16, 1)])
def test_rows_off_the_16_byte_grid(osd, N, V, dtype, shift):
    z, t, u = _inputs(N, V, dtype, seed=V + N + shift)
    u[0], u[N // 2] = 0.0, float(np.nextafter(np.float32(1), np.float32(0)))  # the row's two ends
    store = torch.zeros(N * V + shift, dtype=dtype, device="cuda")
    td = store[shift:].view(N, V)
    td.copy_(t)
    gap = torch.empty(N, device="cuda")
    tok, _ = osd.osd_mixed_sample(z.cuda(), td, u.cuda(), 0.4, temperature=0.9, cdf_gap=gap)
    torch.cuda.synchronize()
    ref, ref_gap = oracle.mixed_sample(z, t, u, 0.4, float(np.float32(0.9)))
    ok = ref_gap >= TIE
    np.testing.assert_array_equal(tok.cpu().numpy()[ok], ref[ok])
    assert np.all(np.abs(gap.cpu().numpy()[ok] - ref_gap[ok]) <= 2e-6)
    assert np.all((tok.cpu().numpy() >= 0) & (tok.cpu().numpy() < V))


# Few rows: 16 and 32 warps a row, at the row counts and lengths where the choice changes.
@pytest.mark.parametrize("N,V,dtype", [
    (1, 6399, torch.bfloat16), (1, 6400, torch.bfloat16), (608, 3200, torch.float32), (609, 3200, torch.float32),
    (3, 65535, torch.bfloat16), (3, 65792, torch.bfloat16), (2, 32897, torch.float32), (5, 102657, torch.bfloat16)])
def test_few_rows(osd, N, V, dtype):
    z, t, u = _inputs(N, V, dtype, seed=3 * V + N)
    u[0], u[N // 2] = 0.0, float(np.nextafter(np.float32(1), np.float32(0)))
    z[0, : V // 2] = float("-inf")  # pieces without mass
    t[0, : V // 2] = float("-inf")
    _check(osd, z, t, u, 0.4, 0.9)
