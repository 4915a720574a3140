"""fp4_momentum_update / fp4_momentum_decode against the oracle: M_t, codes, scales and the
histogram bit for bit, over several steps, with and without stochastic rounding."""
import numpy as np
import pytest
import torch

import oracle
import paper_2607_04422_b200 as fp4
from paper_2607_04422_b200 import workloads
from paper_2607_04422_b200.binding import fp4_root_ns_workspace_layout
from helpers import mismatch_report

pytestmark = pytest.mark.gpu


class GpuState:
    def __init__(self, rows, cols):
        self.codes = torch.zeros((rows, cols // 2), dtype=torch.uint8, device="cuda")
        self.scales = torch.zeros((rows, cols // 16), dtype=torch.int16, device="cuda")

    def load(self, codes, scales):
        self.codes.copy_(torch.from_numpy(codes))
        self.scales.copy_(torch.from_numpy(scales.view(np.int16)))

    def numpy(self):
        return self.codes.cpu().numpy(), self.scales.cpu().numpy().view(np.uint16)


def _step(G_np, st, mu, g_scale=1.0, sr=False, seed=0, want_m=True, want_hist=True):
    G = torch.from_numpy(G_np).cuda()
    M = torch.empty_like(G) if want_m else None
    hist = torch.zeros(8192, dtype=torch.int32, device="cuda") if want_hist else None
    fp4.fp4_momentum_update(G, st.codes, st.scales, M, hist, mu, g_scale,
                            flags=fp4.FP4_MOM_FLAG_SR if sr else 0, seed=seed)
    torch.cuda.synchronize()
    return (M.cpu().numpy() if want_m else None,
            hist.cpu().numpy().view(np.uint32) if want_hist else None)


def _gradient(rows, cols, seed, scale=1.0):
    return (workloads.row_lognormal(rows, cols, seed=seed) * np.float32(scale)).astype(np.float32)


@pytest.mark.parametrize("sr", [False, True])
@pytest.mark.parametrize("shape", [(16, 16), (1, 4096), (48, 272), (300, 1040), (1024, 3072)])
def test_three_steps_bit_exact(shape, sr):
    rows, cols = shape
    st = GpuState(rows, cols)
    oc = np.zeros((rows, cols // 2), np.uint8)
    os_ = np.zeros((rows, cols // 16), np.uint16)
    for t in range(3):
        G = _gradient(rows, cols, seed=10 * t + rows, scale=1.0 + t)
        M, hist = _step(G, st, mu=0.95, g_scale=1.0, sr=sr, seed=77 + t)
        oM, oc, os_, oh = oracle.momentum_update(G, oc, os_, 0.95, 1.0, sr=sr, seed=77 + t)
        c, s = st.numpy()
        assert np.array_equal(M.view(np.uint32), oM.view(np.uint32)), mismatch_report(M, oM)
        assert np.array_equal(s, os_), mismatch_report(s, os_)
        assert np.array_equal(c, oc), mismatch_report(c, oc)
        assert np.array_equal(hist, oh)


def test_ema_form_and_optional_outputs():
    rows, cols = 64, 512
    G = _gradient(rows, cols, seed=3)
    st = GpuState(rows, cols)
    c0, s0 = oracle.momentum_encode(_gradient(rows, cols, seed=4))
    st.load(c0, s0)
    M, hist = _step(G, st, mu=0.9, g_scale=0.1, want_m=False, want_hist=False)
    assert M is None and hist is None
    _, oc, os_, _ = oracle.momentum_update(G, c0, s0, 0.9, 0.1)
    c, s = st.numpy()
    assert np.array_equal(c, oc) and np.array_equal(s, os_)


def _errors_of_both_scales(h):
    """FP64 errors of the nearest-rounding codes of rows h for the scales BF16(amax / 6) and BF16(amax / 4)."""
    grid = np.array([0, 0.5, 1, 1.5, 2, 3, 4, 6])
    amax = np.abs(h).max(axis=1)
    out = []
    for div in (6, 4):
        d = oracle.bf16_bits((amax / np.float32(div)).astype(np.float32)).astype(np.uint32)
        d = (d << 16).view(np.float32).astype(np.float64)[:, None]
        y = np.abs(h) / d
        q = grid[np.abs(y[..., None] - grid).argmin(axis=-1)]
        out.append((((y - q) * d) ** 2).sum(axis=1))
    return out


@pytest.mark.parametrize("scale", [1.0, 2.0 ** -56, 2.0 ** 54, 2.0 ** -90, 2.0 ** 95])
def test_nearly_tied_candidate_scales_take_the_order_of_the_definition(scale):
    """Blocks whose two candidate errors agree to a few parts per million, and neighbours of them on both sides of the tie:
    what the kernel may decide from rounded sums and what it must leave to the definition, in the middle and around both
    ends of the range in which it uses rounded sums.  Far outside all squares underflow or overflow: ties, which keep 6."""
    rng = np.random.default_rng(5)
    H = np.array([[(-1) ** bin(i & j).count("1") for j in range(16)] for i in range(16)], np.float64) / 4
    g = rng.standard_normal((1 << 17, 16)).astype(np.float32)
    e6, e4 = _errors_of_both_scales((g.astype(np.float64) @ H).astype(np.float32))
    close = np.abs(e4 - e6) / np.maximum(e4, e6)
    g = g[np.argsort(close)[:256]]
    assert close[np.argsort(close)[255]] < 2e-2 and close.min() < 1e-4
    # a step along one element that moves the difference of the errors through zero
    blocks = [g]
    for i in (0, 7):
        step = np.zeros_like(g)
        step[:, i] = 2.0 ** -12
        f = lambda x: (lambda a: a[1] - a[0])(_errors_of_both_scales((x.astype(np.float64) @ H).astype(np.float32)))
        lo, hi = g - step * 64, g + step * 64
        assert (np.sign(f(lo)) != np.sign(f(hi))).sum() > 50
        for _ in range(30):                            # bisection in FP32, where the signs differ
            mid = ((lo.astype(np.float64) + hi) / 2).astype(np.float32)
            same = (np.sign(f(mid)) == np.sign(f(lo)))[:, None]
            lo, hi = np.where(same, mid, lo), np.where(same, hi, mid)
        for ulps in (-3, -1, 0, 1, 3):
            b = lo.copy()
            b[:, i] = (b[:, i].view(np.int32) + ulps).view(np.float32)
            blocks.append(b)
    G = (np.concatenate(blocks).reshape(-1, 256) * np.float32(scale)).astype(np.float32)
    st = GpuState(*G.shape)
    _step(G, st, mu=0.0)
    zero = np.zeros((G.shape[0], 128), np.uint8), np.zeros((G.shape[0], 16), np.uint16)
    _, oc, os_, _ = oracle.momentum_update(G, *zero, 0.0, 1.0)
    amax = np.abs((G.reshape(-1, 16).astype(np.float64) @ H).astype(np.float32)).max(axis=1)
    six, four = ((os_.ravel() == oracle.bf16_bits((amax / np.float32(k)).astype(np.float32))).sum() for k in (6, 4))
    if 2.0 ** -60 < scale < 2.0 ** 60:
        assert min(six, four) > 0.2 * amax.size         # both candidates are chosen
        assert scale == 1.0 or amax.min() < 2.0 ** (-55 if scale < 1 else 55) < amax.max()
    else:
        assert six > 0.95 * amax.size
    c, s = st.numpy()
    assert np.array_equal(s, os_), mismatch_report(s, os_)
    assert np.array_equal(c, oc), mismatch_report(c, oc)


@pytest.mark.parametrize("sr", [False, True])
@pytest.mark.parametrize("scale", [1.0, 2.0 ** -54, 2.0 ** -57, 2.0 ** 53, 2.0 ** 56])
def test_blocks_of_one_magnitude_and_their_exact_ties(scale, sr):
    """Constant blocks and blocks of one element: in the transformed domain one value beside zeros, and sixteen equal magnitudes.
    A third of them have the same values with both scales, some lie midway between the values of both: exact ties, which keep 6
    without the sums of the definition.  Their neighbours on both sides are not ties.  Also around the ends of the range in
    which the kernel compares scaled errors (2^-55, 2^55)."""
    amax = 1 + np.arange(2048) / 2048
    amax = np.concatenate([amax, np.nextafter(amax.astype(np.float32), np.float32(2)), np.nextafter(amax.astype(np.float32), np.float32(0))])
    amax = amax.astype(np.float32)
    d6, d4 = ((oracle.bf16_bits((amax / np.float32(k)).astype(np.float32)).astype(np.uint32) << 16).view(np.float32).astype(np.float64)
              for k in (6, 4))
    e6, e4 = np.abs(amax - 6 * d6), np.abs(amax - 4 * d4)
    assert (d4 == 1.5 * d6).sum() > 500 and ((d4 != 1.5 * d6) & (e6 == e4)).sum() > 20
    assert (e6 < e4).sum() > 1000 and (e4 < e6).sum() > 1000
    amax = amax * np.float32(scale)
    G = np.zeros((2, amax.size, 16), np.float32)
    G[0] = amax[:, None] / 4                                    # h = amax, 0, 0, ...
    G[1, np.arange(amax.size), np.arange(amax.size) % 16] = 4 * amax   # |h| = amax
    G = G.reshape(-1, 256)
    st = GpuState(*G.shape)
    _step(G, st, mu=0.0, sr=sr, seed=9)
    zero = np.zeros((G.shape[0], 128), np.uint8), np.zeros((G.shape[0], 16), np.uint16)
    _, oc, os_, _ = oracle.momentum_update(G, *zero, 0.0, 1.0, sr=sr, seed=9)
    c, s = st.numpy()
    assert np.array_equal(s, os_), mismatch_report(s, os_)
    assert np.array_equal(c, oc), mismatch_report(c, oc)


@pytest.mark.parametrize("nonzeros", [2, 3, 4])
def test_blocks_of_few_magnitudes(nonzeros):
    """Sparse blocks, five steps of the same gradient: states that settle on few magnitudes and tie often."""
    rng = np.random.default_rng(nonzeros)
    G = np.zeros((4096, 16), np.float32)
    for _ in range(nonzeros):
        G[np.arange(4096), rng.integers(0, 16, 4096)] = rng.integers(-64, 65, 4096)
    G = G.reshape(-1, 256)
    st = GpuState(*G.shape)
    oc, os_ = np.zeros((256, 128), np.uint8), np.zeros((256, 16), np.uint16)
    for _ in range(5):
        _step(G, st, mu=0.875, g_scale=0.125)
        _, oc, os_, _ = oracle.momentum_update(G, oc, os_, 0.875, 0.125)
        c, s = st.numpy()
        assert np.array_equal(s, os_), mismatch_report(s, os_)
        assert np.array_equal(c, oc), mismatch_report(c, oc)


def test_ties_zero_blocks_and_extreme_magnitudes():
    f = np.float32
    H4 = oracle.hadamard16  # only to place chosen values in the transformed domain
    rng = np.random.default_rng(1)
    rows, cols = 32, 256
    G = np.zeros((rows, cols), f)
    mids = np.array([0.25, 0.75, 1.25, 1.75, 2.5, 3.5, 5.0, 6.0, 4.0, 3.0, 0.0, 0.5, 1.0, 1.5, 2.0], f)
    for r in range(rows):
        for b in range(cols // 16):
            h = rng.choice(np.concatenate([mids, -mids]), 16).astype(f)
            h[rng.integers(16)] = [6.0, 4.0, 6.0 * 1.00390625, 5.0][(r + b) % 4]
            h = h * f(2.0) ** int(rng.integers(-30, 30))
            G[r, b * 16:(b + 1) * 16] = H4(h)      # the transform is its own inverse
    G[3, 32:48] = 0
    G[4, 0:16] = f(1e-42)                          # denormals
    G[5, 16:32] = f(1e37) * np.sign(rng.standard_normal(16)).astype(f)   # sums stay finite
    G[6, 0:16] = 0
    G[6, 5] = f(-1e-30)
    for sr in (False, True):
        st = GpuState(rows, cols)
        M, hist = _step(G, st, mu=0.5, sr=sr, seed=9)
        oM, oc, os_, oh = oracle.momentum_update(G, np.zeros((rows, cols // 2), np.uint8),
                                                 np.zeros((rows, cols // 16), np.uint16), 0.5, sr=sr, seed=9)
        c, s = st.numpy()
        assert np.array_equal(M.view(np.uint32), oM.view(np.uint32))
        assert np.array_equal(s, os_), mismatch_report(s, os_)
        assert np.array_equal(c, oc), mismatch_report(c, oc)
        assert np.array_equal(hist, oh)
        # second step from that state: the decode of every such block
        G2 = np.zeros_like(G)
        M2, _ = _step(G2, st, mu=1.0, sr=sr, seed=10)
        oM2, _, _, _ = oracle.momentum_update(G2, oc, os_, 1.0, sr=sr, seed=10)
        assert np.array_equal(M2.view(np.uint32), oM2.view(np.uint32))


def test_decode_entry_point():
    rows, cols = 96, 784
    c0, s0 = oracle.momentum_encode(_gradient(rows, cols, seed=12))
    st = GpuState(rows, cols)
    st.load(c0, s0)
    M = torch.empty((rows, cols), dtype=torch.float32, device="cuda")
    fp4.fp4_momentum_decode(st.codes, st.scales, M)
    torch.cuda.synchronize()
    assert np.array_equal(M.cpu().numpy().view(np.uint32), oracle.momentum_decode(c0, s0).view(np.uint32))
    c, s = st.numpy()
    assert np.array_equal(c, c0) and np.array_equal(s, s0)


def test_full_size_sampled_rows_and_histogram():
    # the benchmark's size: rows checked one by one against the oracle, the histogram against the
    # kernel's own M_t
    rows, cols = 8192, 8192
    gen = torch.Generator(device="cuda").manual_seed(5)
    G = torch.randn((rows, cols), generator=gen, device="cuda", dtype=torch.float32)
    G *= torch.exp(0.5 * torch.randn((rows, 1), generator=gen, device="cuda"))
    st = GpuState(rows, cols)
    M = torch.empty_like(G)
    hist = torch.zeros(8192, dtype=torch.int32, device="cuda")
    for t in range(2):
        prev_c, prev_s = st.codes.clone(), st.scales.clone()
        hist.zero_()
        fp4.fp4_momentum_update(G, st.codes, st.scales, M, hist, 0.95, 1.0, flags=fp4.FP4_MOM_FLAG_SR, seed=t)
    torch.cuda.synchronize()
    assert int(hist.sum().item()) == rows * cols
    bins = (M.view(torch.int32) & 0x7FFFFFFF) >> 18
    want = torch.bincount(bins.flatten().long(), minlength=8192)
    assert torch.equal(want.to(torch.int32), hist)
    # without stochastic rounding any row can be checked alone; with it the random stream is
    # numbered by matrix position, so the leading rows are
    head = 8
    oM, oc, os_, _ = oracle.momentum_update(G[:head].cpu().numpy(), prev_c[:head].cpu().numpy(),
                                            prev_s[:head].cpu().numpy().view(np.uint16), 0.95, 1.0, sr=True, seed=1)
    assert np.array_equal(M[:head].cpu().numpy().view(np.uint32), oM.view(np.uint32))
    assert np.array_equal(st.codes[:head].cpu().numpy(), oc)
    assert np.array_equal(st.scales[:head].cpu().numpy().view(np.uint16), os_)
    idx = torch.tensor(np.random.default_rng(0).choice(rows, 24, replace=False), device="cuda")
    Gs = G[idx].cpu().numpy()
    pc, ps = prev_c[idx].cpu().numpy(), prev_s[idx].cpu().numpy().view(np.uint16)
    st2_c, st2_s = prev_c.clone(), prev_s.clone()
    fp4.fp4_momentum_update(G, st2_c, st2_s, M, None, 0.95, 1.0)
    torch.cuda.synchronize()
    oM, oc, os_, _ = oracle.momentum_update(Gs, pc, ps, 0.95, 1.0)
    assert np.array_equal(M[idx].cpu().numpy().view(np.uint32), oM.view(np.uint32))
    assert np.array_equal(st2_c[idx].cpu().numpy(), oc)
    assert np.array_equal(st2_s[idx].cpu().numpy().view(np.uint16), os_)


def test_argument_errors():
    G = torch.zeros((16, 24), dtype=torch.float32, device="cuda")
    c = torch.zeros((16, 12), dtype=torch.uint8, device="cuda")
    s = torch.zeros((16, 2), dtype=torch.int16, device="cuda")
    with pytest.raises(fp4.Fp4Error):
        fp4.fp4_momentum_update(G, c, s, None, None, 0.9)            # cols not a multiple of 16
    G = torch.zeros((16, 32), dtype=torch.float32, device="cuda")
    c = torch.zeros((16, 16), dtype=torch.uint8, device="cuda")
    with pytest.raises(fp4.Fp4Error):
        fp4.fp4_momentum_update(G, c, s, None, None, 0.9, flags=4)   # unknown flag
    with pytest.raises(fp4.Fp4Error):
        fp4.fp4_momentum_update(G.flatten()[1:].reshape(1, -1)[:, :16], c, s, None, None, 0.9)  # misaligned
    with pytest.raises(fp4.Fp4Error):
        fp4.fp4_momentum_update(G.flatten()[4:].reshape(1, -1)[:, :16], c, s, None, None, 0.9)  # 16 but not 32 bytes


def _ns(G, steps=2, top_hist=None):
    m, n = G.shape
    out = torch.full((m, n), float("nan"), device="cuda")
    ws = torch.empty(fp4.fp4_root_ns_workspace_bytes(m, n, steps, 0), dtype=torch.uint8, device="cuda")
    p = fp4.NsParams.make(top_hist=top_hist)
    fp4.fp4_root_ns(G, out, steps, p, ws)
    assert fp4.fp4_last_device_status(ws) == 0
    return out


@pytest.mark.parametrize("shape", [(256, 512), (1024, 384), (400, 1136)])
def test_momentum_histogram_feeds_the_clip(shape):
    # M_t and its histogram from the momentum step; the Newton-Schulz step that takes the
    # histogram must give exactly what it gives when it counts M_t itself, and the oracle chain
    # (momentum step, then Root step) must agree with the GPU chain
    rows, cols = shape
    G = _gradient(rows, cols, seed=21)
    st = GpuState(rows, cols)
    c0, s0 = oracle.momentum_encode(_gradient(rows, cols, seed=22))
    st.load(c0, s0)
    Gd = torch.from_numpy(G).cuda()
    M = torch.empty_like(Gd)
    hist = torch.zeros(8192, dtype=torch.int32, device="cuda")
    fp4.fp4_momentum_update(Gd, st.codes, st.scales, M, hist, 0.95, 1.0)
    ref = _ns(M)
    got = _ns(M, top_hist=[hist])
    torch.cuda.synchronize()
    assert torch.equal(ref, got)
    assert int(hist.abs().sum().item()) == 0          # consumed
    oM, _, _, _ = oracle.momentum_update(G, c0, s0, 0.95, 1.0)
    assert np.array_equal(M.cpu().numpy().view(np.uint32), oM.view(np.uint32))
    want = oracle.root_ns(oM, 2)
    err = np.linalg.norm(got.cpu().numpy() - want) / np.linalg.norm(want)
    assert err < 2e-3, err


def test_momentum_histograms_in_a_batched_call():
    shapes = [(256, 512), (256, 512), (512, 256), (384, 384), (256, 512)]
    Ms, hists, outs_ref = [], [], []
    for i, (r, c) in enumerate(shapes):
        Gd = torch.from_numpy(_gradient(r, c, seed=30 + i)).cuda()
        st = GpuState(r, c)
        M = torch.empty_like(Gd)
        h = torch.zeros(8192, dtype=torch.int32, device="cuda")
        fp4.fp4_momentum_update(Gd, st.codes, st.scales, M, h, 0.9, 1.0)
        Ms.append(M)
        hists.append(h if i != 1 else None)           # one matrix of a group counts for itself
        outs_ref.append(_ns(M, steps=3))
    outs = [torch.empty_like(M) for M in Ms]
    ws = torch.empty(fp4.fp4_root_ns_batched_workspace_bytes(shapes, 3, 0), dtype=torch.uint8, device="cuda")
    fp4.fp4_root_ns_batched(Ms, outs, 3, fp4.NsParams.make(top_hist=hists), ws)
    assert fp4.fp4_last_device_status(ws) == 0
    for a, b in zip(outs, outs_ref):
        assert torch.equal(a, b)
    for h in hists:
        if h is not None:
            assert int(h.abs().sum().item()) == 0


@pytest.mark.parametrize("shape", [(256, 512), (1136, 400), (128, 57088)])
def test_momentum_histogram_is_consumed_whichever_way_the_clip_level_is_found(shape):
    """The same counters over three steps: an all-zero momentum and one of few values (more elements in the clip's bin than its
    candidate list takes), then a dense one.  After every step the counters are zero, and clip level and result are those of the
    step that counts for itself.  One cooperative prologue launch for the first two shapes, several launches for the last."""
    rows, cols = shape
    rng = np.random.default_rng(rows)
    grads = [np.zeros(shape, np.float32), rng.choice([-1.0, 0.5, 2.0], shape).astype(np.float32), _gradient(rows, cols, seed=4)]
    st = GpuState(rows, cols)
    M = torch.empty(shape, device="cuda")
    hist = torch.zeros(8192, dtype=torch.int32, device="cuda")
    ws = torch.empty(fp4.fp4_root_ns_workspace_bytes(rows, cols, 1), dtype=torch.uint8, device="cuda")
    lay = fp4_root_ns_workspace_layout(rows, cols, 1)

    def step(top_hist):
        out = torch.full(shape, float("nan"), device="cuda")
        fp4.fp4_root_ns(M, out, 1, fp4.NsParams.make(top_hist=top_hist), ws)
        assert fp4.fp4_last_device_status(ws) == 0
        return out, ws[lay.scalars:lay.scalars + 4096].cpu().numpy().view(np.float32)[lay.idx_tau]

    for g in grads:
        fp4.fp4_momentum_update(torch.from_numpy(g).cuda(), st.codes, st.scales, M, hist, 0.95, 1.0)
        assert int(hist.sum().item()) == rows * cols
        got, tau = step([hist])
        assert int(hist.abs().sum().item()) == 0
        a = M.abs().flatten()
        assert tau == a.kthvalue(-(-99 * a.numel() // 100)).values.item()
        ref, ref_tau = step(None)
        assert tau == ref_tau and torch.equal(got, ref)


def test_optimizer_chain_in_a_cuda_graph():
    """Momentum step, Root step with the histogram handed over and a packed AdamW step only
    enqueue kernels on their stream: the chain is captured once and replayed on new gradients."""
    rows, cols = 256, 512
    n = rows * cols
    G = torch.empty((rows, cols), device="cuda")
    Gb = torch.empty(n, dtype=torch.bfloat16, device="cuda")
    st = GpuState(rows, cols)
    M = torch.empty_like(G)
    hist = torch.zeros(8192, dtype=torch.int32, device="cuda")
    out = torch.empty_like(G)
    ws = torch.empty(fp4.fp4_root_ns_workspace_bytes(rows, cols, 3), dtype=torch.uint8, device="cuda")
    W = torch.zeros(n, dtype=torch.bfloat16, device="cuda")
    mc = torch.zeros(n // 2, dtype=torch.uint8, device="cuda"); ms = torch.zeros(n // 16, dtype=torch.int16, device="cuda")
    vc = torch.zeros(n // 2, dtype=torch.uint8, device="cuda"); vs = torch.zeros(n // 16, dtype=torch.int16, device="cuda")
    vm = torch.zeros(n // 256, dtype=torch.int16, device="cuda")
    prm = fp4.NsParams.make(top_hist=[hist])

    def chain(stream=None):
        fp4.fp4_momentum_update(G, st.codes, st.scales, M, hist, 0.95, 1.0, stream=stream)
        fp4.fp4_root_ns(M, out, 3, prm, ws, stream)
        fp4.fp4_adamw_update(W, Gb, mc, ms, vc, vs, vm, lr=1e-3, step=1, stream=stream)

    G.copy_(torch.from_numpy(_gradient(rows, cols, seed=50)))
    Gb.copy_(G.flatten().to(torch.bfloat16))
    chain()                                   # per-device set-up happens outside the capture
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        chain(torch.cuda.current_stream())
    # oracle mirror of the replays, starting from the states the direct call and the capture left
    # (a capture does not execute anything)
    oc, os_ = st.numpy()
    oW = W.view(torch.int16).cpu().numpy().view(np.uint16)
    ost = (mc.cpu().numpy(), ms.cpu().numpy().view(np.uint16), vc.cpu().numpy(), vs.cpu().numpy().view(np.uint16),
           vm.cpu().numpy().view(np.uint16))
    for rep in range(2):
        g_np = _gradient(rows, cols, seed=60 + rep)
        G.copy_(torch.from_numpy(g_np))
        Gb.copy_(G.flatten().to(torch.bfloat16))
        graph.replay()
        torch.cuda.synchronize()
        assert fp4.fp4_last_device_status(ws) == 0
        oM, oc, os_, _ = oracle.momentum_update(g_np, oc, os_, 0.95, 1.0)
        assert np.array_equal(M.cpu().numpy().view(np.uint32), oM.view(np.uint32))
        c, s = st.numpy()
        assert np.array_equal(c, oc) and np.array_equal(s, os_)
        want = oracle.root_ns(oM, 3)
        err = np.linalg.norm(out.cpu().numpy() - want) / np.linalg.norm(want)
        assert err < 2e-3, err
        assert int(hist.abs().sum().item()) == 0
        gb = Gb.view(torch.int16).cpu().numpy().view(np.uint16)
        oW, ost, _, _ = oracle.adamw_update(oW, gb, ost, lr=1e-3, step=1)
        assert np.array_equal(W.view(torch.int16).cpu().numpy().view(np.uint16), oW)
