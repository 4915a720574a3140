"""fp4_quantize against the oracle: codes, scales and tensor scale bit for bit."""
import time

import numpy as np
import pytest
import torch

import oracle
import paper_2607_04422_b200 as fp4
from paper_2607_04422_b200 import workloads
from paper_2607_04422_b200.binding import FP4_FLAG_FOUR_SIX, FP4_FLAG_RHT
from helpers import mismatch_report, sf_from_atoms

pytestmark = pytest.mark.gpu


def _run(x_np, flags=0):
    rows, cols = x_np.shape
    x = torch.from_numpy(x_np).cuda()
    codes = torch.empty((rows, cols // 2), dtype=torch.uint8, device="cuda")
    scales = torch.zeros(fp4.fp4_scale_bytes(rows, cols), dtype=torch.uint8, device="cuda")
    ts = torch.zeros(1, dtype=torch.float32, device="cuda")
    fp4.fp4_quantize(x, codes, scales, ts, flags=flags)
    torch.cuda.synchronize()
    return codes.cpu().numpy(), sf_from_atoms(scales.cpu().numpy(), rows, cols // 16), float(ts.item())


def _compare(x_np):
    c, s, sg = _run(x_np)
    oc, os_, osg = oracle.quantize(x_np)
    assert np.float32(sg) == np.float32(osg)
    assert np.array_equal(s, os_), mismatch_report(s, os_)
    assert np.array_equal(c, oc), mismatch_report(c, oc)


def test_ties_saturation_and_signed_zero():
    # every E2M1 midpoint and its neighbours, E4M3 midpoints as block maxima, zeros
    f = np.float32
    mids = np.array([0.25, 0.75, 1.25, 1.75, 2.5, 3.5, 5.0], f)
    pts = np.concatenate([mids, np.nextafter(mids, f(0)), np.nextafter(mids, f(10)),
                          np.array([0, 0.5, 1, 1.5, 2, 3, 4, 6, 1e-8, 6.0], f)])
    pts = np.concatenate([pts, -pts])
    x = np.zeros((128, 128), f)
    rng = np.random.default_rng(0)
    for r in range(128):
        for b in range(8):
            blk = rng.choice(pts, 16)
            # block maximum on or next to an E4M3 rounding boundary in some rows
            top = [6.0, 6.375, 6.75, 6.0 * 1.0625, np.nextafter(f(6.375), f(7)), 5.9][(r + b) % 6]
            blk[rng.integers(16)] = top
            x[r, b * 16:(b + 1) * 16] = blk
    x[5, 16:32] = 0  # an all-zero block
    x[0, 0] = 2688.0  # tensor amax 2688 -> s_g = 1 exactly, so the ties above are hit exactly
    _compare(x * f(0.37))
    _compare(x)


@pytest.mark.parametrize("gen,shape", [
    (workloads.gaussian, (256, 512)),
    (workloads.row_lognormal, (384, 1024)),
    (workloads.lowrank_outliers, (128, 2048)),
    (workloads.gradient_like, (1024, 640)),
])
def test_workloads_bit_exact(gen, shape):
    _compare(gen(*shape, seed=3))


def test_all_zero_tensor():
    c, s, sg = _run(np.zeros((128, 128), np.float32))
    assert sg == 1.0 and not c.any() and not s.any()


def test_large_tensor_sampled_rows():
    # a tensor larger than L2; the oracle checks a sample of rows
    x = workloads.gaussian(4096, 8192, seed=5)
    c, s, sg = _run(x)
    assert np.float32(sg) == np.float32(np.abs(x).max() / np.float32(2688))
    rows = np.random.default_rng(0).choice(4096, 64, replace=False)
    oc, os_, _ = oracle.quantize(x[rows], s_g=sg)
    assert np.array_equal(c[rows], oc) and np.array_equal(s[rows], os_)


@pytest.mark.parametrize("rht,four_six", [(True, False), (False, True), (True, True)])
@pytest.mark.parametrize("gen,shape", [
    (workloads.gaussian, (256, 512)),
    (workloads.row_lognormal, (384, 1024)),
    (workloads.gradient_like, (128, 4224)),     # a row is longer than one thread block covers
])
def test_paper_faithful_options_bit_exact(gen, shape, rht, four_six):
    """Random Hadamard transform and adaptive 4/6 (Section 3.4): the transform's butterfly
    order and the order of the error sums are part of the definition, so codes, block
    scales and the tensor scale agree bit for bit."""
    x = gen(*shape, seed=5)
    mask = oracle.rht_mask(17, 3) if rht else 0
    flags = (FP4_FLAG_RHT | (mask << 16) if rht else 0) | (FP4_FLAG_FOUR_SIX if four_six else 0)
    c, s, sg = _run(x, flags)
    oc, os_, osg = oracle.quantize(x, rht=rht, mask=mask, four_six=four_six)
    assert np.float32(sg) == np.float32(osg)
    assert np.array_equal(s, os_), mismatch_report(s, os_)
    assert np.array_equal(c, oc), mismatch_report(c, oc)
    if four_six:
        base = oracle.quantize(x, rht=rht, mask=mask)
        assert (s != base[1]).mean() > 0.05      # the 4-mapping is really taken


def test_paper_faithful_options_edge_blocks():
    """Blocks whose two candidate encodings tie or underflow."""
    x = np.zeros((128, 128), np.float32)
    x[0, :16] = [6, 3, 1.5, 0, 0, 0, 0, 0, 0, 0, 0, 0, 0, 0, 0, 0]        # tie: keeps the 6-mapping
    x[1, :16] = [4, 3, 2, 1, 0.5, 0, 0, 0, 0, 0, 0, 0, 0, 0, 0, -4]       # the 4-mapping is exact
    x[2, :16] = 1e-9                                                       # block scale underflows to 0
    x[3, 16:32] = np.float32(2688.0)                                       # sets the tensor scale to 1
    x[4, :16] = 5.0 / 1024                                                  # 6-scale 0, 4-scale the smallest subnormal
    c, s, sg = _run(x, FP4_FLAG_FOUR_SIX)
    oc, os_, osg = oracle.quantize(x, four_six=True)
    assert sg == osg == 1.0
    assert np.array_equal(s, os_), mismatch_report(s, os_)
    assert np.array_equal(c, oc), mismatch_report(c, oc)
    assert s[0, 0] == 0x38 and s[1, 0] == 0x38 and s[2, 0] == 0 and s[4, 0] == 1


def test_argument_errors():
    x = torch.zeros((128, 128), device="cuda")
    codes = torch.empty((128, 64), dtype=torch.uint8, device="cuda")
    scales = torch.zeros(1024, dtype=torch.uint8, device="cuda")
    ts = torch.zeros(1, device="cuda")
    with pytest.raises(fp4.Fp4Error) as e:
        fp4.fp4_quantize(torch.zeros((100, 128), device="cuda"), codes, scales, ts)
    assert e.value.code == 2
    with pytest.raises(fp4.Fp4Error) as e:
        fp4.fp4_quantize(x, codes, scales, ts, flags=7)
    assert e.value.code == 1
    with pytest.raises(fp4.Fp4Error) as e:       # sign bits without the transform flag
        fp4.fp4_quantize(x, codes, scales, ts, flags=FP4_FLAG_FOUR_SIX | (0x1234 << 16))
    assert e.value.code == 1


def _errors_of_both_scales(x, sg):
    """FP64 errors of the nearest-rounding codes of blocks x for the scales E4M3(amax / 6 sg) and E4M3(amax / 4 sg)."""
    grid = np.array([0, 0.5, 1, 1.5, 2, 3, 4, 6])
    amax = np.abs(x).max(axis=1).astype(np.float64)
    out = []
    for div in (6, 4):
        t = amax / (div * float(sg))
        ulp = 2.0 ** (np.floor(np.log2(np.maximum(t, 2.0 ** -6))) - 3)
        d = (np.rint(t / ulp) * ulp * float(sg))[:, None]
        y = np.abs(x) / d
        q = grid[np.abs(y[..., None] - grid).argmin(axis=-1)]
        out.append((((y - q) * d) ** 2).sum(axis=1))
    return out


@pytest.mark.parametrize("sg", [1.0, 1.37, 1.37 * 2.0 ** -47, 1.37 * 2.0 ** -49, 1.37 * 2.0 ** 59, 1.37 * 2.0 ** 61])
def test_nearly_tied_scales_take_the_order_of_the_definition(sg):
    """4/6 without the transform: blocks whose two errors agree to a few units in the last place, and exact ties (equal magnitudes,
    scales with a ratio of 1.5), inside and on both sides of the range in which the kernel decides from rounded sums."""
    rng = np.random.default_rng(3)
    sg = np.float32(sg)
    g = (rng.standard_normal((1 << 16, 16)) * np.exp2(rng.uniform(-2, 9, (1 << 16, 1)))).astype(np.float32) * sg
    e6, e4 = _errors_of_both_scales(g, sg)
    close = np.abs(e4 - e6) / np.maximum(e4, e6)
    g = g[np.argsort(close + (close == 0))[:256]]
    blocks = [g]
    for i in (0, 7):
        step = np.zeros_like(g)
        step[:, i] = np.abs(g).max(axis=1) * 2.0 ** -6
        f = lambda x: (lambda a: a[1] - a[0])(_errors_of_both_scales(x, sg))
        lo, hi = g - step, g + step
        assert (np.sign(f(lo)) != np.sign(f(hi))).sum() > 50
        for _ in range(30):                            # bisection in FP32, where the signs differ
            mid = ((lo.astype(np.float64) + hi) / 2).astype(np.float32)
            same = (np.sign(f(mid)) == np.sign(f(lo)))[:, None]
            lo, hi = np.where(same, mid, lo), np.where(same, hi, mid)
        for ulps in (-3, -1, 0, 1, 3):
            b = lo.copy()
            b[:, i] = (b[:, i].view(np.int32) + ulps).view(np.float32)
            blocks.append(b)
    one = np.where(rng.random((512, 16)) < 0.5, 0, rng.choice([-1.0, 1.0], (512, 16)))
    blocks.append((one * rng.uniform(1, 16, (512, 1))).astype(np.float32) * sg)
    tiny = rng.standard_normal((512, 16)) * np.exp2(rng.uniform(-12, -6, (512, 1)))   # scale bytes in the subnormals, and zero
    blocks.append(tiny.astype(np.float32) * sg)
    x = np.concatenate(blocks)
    x = np.concatenate([x, np.zeros((-len(x) % 1024, 16), np.float32)]).reshape(-1, 128)
    x[-1, -1] = np.float32(2688.0) * sg                # makes sg the tensor scale
    c, s, got = _run(x, FP4_FLAG_FOUR_SIX)
    oc, os_, osg = oracle.quantize(x, four_six=True)
    assert np.float32(got) == np.float32(osg) == sg
    assert np.array_equal(s, os_), mismatch_report(s, os_)
    assert np.array_equal(c, oc), mismatch_report(c, oc)


@pytest.mark.parametrize("flags", [0, FP4_FLAG_RHT | FP4_FLAG_FOUR_SIX])
@pytest.mark.parametrize("shape", [(128, 128), (128, 384), (640, 2432), (128, 56832), (128, 56960)])
def test_single_launch_quantiser_at_its_limits(shape, flags):
    """Tensors that fit the shared memories of all SMs are quantised in one launch: fewer units than SMs, a partial last
    round, the largest on 148 SMs (6 units in each of 4 groups), and the first size beyond; twice the same on
    dirty outputs."""
    rows, cols = shape
    x_np = workloads.row_lognormal(rows, cols, seed=cols)
    mask = 0x5A3C if flags else 0
    x = torch.from_numpy(x_np).cuda()
    oc, os_, osg = oracle.quantize(x_np, rht=True, mask=mask, four_six=True) if flags else oracle.quantize(x_np)
    for _ in range(2):
        codes = torch.full((rows, cols // 2), 0xEE, dtype=torch.uint8, device="cuda")
        scales = torch.full((fp4.fp4_scale_bytes(rows, cols),), 0xEE, dtype=torch.uint8, device="cuda")
        ts = torch.full((1,), float("nan"), device="cuda")
        before = fp4.fp4_kernel_launches()
        fp4.fp4_quantize(x, codes, scales, ts, flags=flags | mask << 16)
        assert fp4.fp4_kernel_launches() - before == (3 if shape == (128, 56960) else 1)
        assert np.float32(ts.item()) == np.float32(osg)
        got = sf_from_atoms(scales.cpu().numpy(), rows, cols // 16)
        assert np.array_equal(got, os_), mismatch_report(got, os_)
        assert np.array_equal(codes.cpu().numpy(), oc), mismatch_report(codes.cpu().numpy(), oc)


@pytest.mark.parametrize("flags", [0, FP4_FLAG_RHT | FP4_FLAG_FOUR_SIX])
@pytest.mark.parametrize("offset", [0, 4, 8])
@pytest.mark.parametrize("shape,scale", [((1792, 4224), 1.0), ((57088, 128), 1.0), ((1792, 4224), 2.0 ** -75)])
def test_two_pass_quantiser_on_every_alignment(shape, scale, offset, flags):
    """Tensors beyond the single launch: on 32-byte boundaries (256-bit loads) and only on 16-byte ones, a row of one and a bit
    thread blocks and of half a warp, a tensor scale below 2^-60 (plain operations)."""
    rows, cols = shape
    x_np = workloads.row_lognormal(rows, cols, seed=rows) * np.float32(scale)
    mask = 0xA5C3 if flags else 0
    store = torch.empty(rows * cols + 8, device="cuda")
    x = store[offset:offset + rows * cols].view(rows, cols)
    assert x.data_ptr() % 32 == offset * 4 % 32
    x.copy_(torch.from_numpy(x_np))
    oc, os_, osg = oracle.quantize(x_np, rht=True, mask=mask, four_six=True) if flags else oracle.quantize(x_np)
    codes = torch.full((rows, cols // 2), 0xEE, dtype=torch.uint8, device="cuda")
    scales = torch.full((fp4.fp4_scale_bytes(rows, cols),), 0xEE, dtype=torch.uint8, device="cuda")
    ts = torch.full((1,), float("nan"), device="cuda")
    fp4.fp4_quantize(x, codes, scales, ts, flags=flags | mask << 16)
    assert np.float32(ts.item()) == np.float32(osg)
    got = sf_from_atoms(scales.cpu().numpy(), rows, cols // 16)
    assert np.array_equal(got, os_), mismatch_report(got, os_)
    assert np.array_equal(codes.cpu().numpy(), oc), mismatch_report(codes.cpu().numpy(), oc)


@pytest.mark.parametrize("scale", [1.0, 1e-41])    # the second: a tensor scale of a few units of 2^-149
@pytest.mark.parametrize("shape", [(128, 128), (1024, 1152), (1152, 2688)])
def test_single_launch_quantiser_waits_for_no_word_that_it_overwrites(shape, scale):
    """Blocks of the single launch go on to write scales while others may still be at its last barrier.  Zero scale bytes
    throughout the first two atoms - whatever the blocks could share there - must stall nobody: a wait that nothing ends takes
    two seconds to give up, 200 calls take a few milliseconds."""
    rows, cols = shape
    x_np = workloads.gaussian(rows, cols, seed=cols) * np.float32(scale)
    # below 2^-128 the reciprocal of a block's scale is infinite: 0 times it is a NaN, whose code is nowhere defined
    x_np[x_np == 0] = scale
    x_np[:128, :128] = 0
    if shape == (128, 128):
        x_np[0, :16] = scale
    x = torch.from_numpy(x_np).cuda()
    codes = torch.empty((rows, cols // 2), dtype=torch.uint8, device="cuda")
    scales = torch.empty(fp4.fp4_scale_bytes(rows, cols), dtype=torch.uint8, device="cuda")
    ts = torch.empty(1, device="cuda")
    fp4.fp4_quantize(x, codes, scales, ts)
    torch.cuda.synchronize()
    t0 = time.monotonic()
    for _ in range(200):
        fp4.fp4_quantize(x, codes, scales, ts)
    torch.cuda.synchronize()
    assert time.monotonic() - t0 < 1.0
    oc, os_, osg = oracle.quantize(x_np)
    assert np.float32(ts.item()) == np.float32(osg)
    assert np.array_equal(sf_from_atoms(scales.cpu().numpy(), rows, cols // 16), os_)
    assert np.array_equal(codes.cpu().numpy(), oc)


@pytest.mark.parametrize("scale", [1.0, 1e-41])
@pytest.mark.parametrize("shape", [(128, 128), (1152, 2688)])
def test_single_launch_quantiser_reports_that_it_gave_up(shape, scale):
    """Barriers that expect a block which is not launched give up after the limit, and the tensor scale says so; the
    next call on the same buffers is whole."""
    rows, cols = shape
    x_np = workloads.gaussian(rows, cols, seed=2) * np.float32(scale)
    x = torch.from_numpy(x_np).cuda()
    codes = torch.empty((rows, cols // 2), dtype=torch.uint8, device="cuda")
    scales = torch.empty(fp4.fp4_scale_bytes(rows, cols), dtype=torch.uint8, device="cuda")
    ts = torch.ones(1, device="cuda")
    fp4.fp4_selftest_quantize_wait(x, codes, scales, ts, 200)
    assert np.isnan(ts.item())
    fp4.fp4_quantize(x, codes, scales, ts)
    oc, os_, osg = oracle.quantize(x_np)
    assert np.float32(ts.item()) == np.float32(osg)
    assert np.array_equal(sf_from_atoms(scales.cpu().numpy(), rows, cols // 16), os_)


@pytest.mark.parametrize("flags", [0, FP4_FLAG_RHT | 0x2D5A0000, FP4_FLAG_FOUR_SIX, FP4_FLAG_RHT | FP4_FLAG_FOUR_SIX | 0x2D5A0000])
@pytest.mark.parametrize("shape,offset", [((2816, 2688), 0), ((4224, 5760), 0), ((4224, 5760), 4)])
def test_blocks_of_the_second_pass_wait_for_the_maximum_of_the_whole_tensor(shape, offset, flags):
    """The second pass starts at the tensor's end while blocks of the first still run: wherever the largest magnitude lies, whoever
    reads it last, the last rows have its scale."""
    rows, cols = shape
    gen = torch.Generator(device="cuda").manual_seed(7)
    buf = torch.randn(rows * cols + 8, device="cuda", generator=gen)
    x = buf[offset:offset + rows * cols].view(shape)                 # 4: on a 16-byte, not on a 32-byte boundary
    codes = torch.empty((rows, cols // 2), dtype=torch.uint8, device="cuda")
    scales = torch.empty(fp4.fp4_scale_bytes(rows, cols), dtype=torch.uint8, device="cuda")
    ts = torch.empty(1, device="cuda")
    widen = np.float32(4 if flags & FP4_FLAG_RHT else 1)
    sg = widen * np.float32(64) / np.float32(2688)
    last = x[-128:].cpu().numpy()
    want_codes, want_scales, _ = oracle.quantize(last, s_g=sg, rht=bool(flags & FP4_FLAG_RHT), mask=flags >> 16,
                                                 four_six=bool(flags & FP4_FLAG_FOUR_SIX))
    rng = np.random.default_rng(1)
    for at in rng.integers(0, (rows - 128) * cols, 48):
        keep = x.view(-1)[at].clone()
        x.view(-1)[at] = 64.0
        fp4.fp4_quantize(x, codes, scales, ts, flags=flags)
        x.view(-1)[at] = keep
        assert np.float32(ts.item()) == sg
        got = sf_from_atoms(scales[-128 * (cols // 16):].cpu().numpy(), 128, cols // 16)
        assert np.array_equal(got, want_scales), (int(at), mismatch_report(got, want_scales))
        assert np.array_equal(codes[-128:].cpu().numpy(), want_codes), int(at)


def test_long_rows_take_no_longer_than_short_ones():
    # the second pass reads from the tensor's end, where the L2 still holds it, also where a row takes several thread blocks: measured 0.99
    # times the time of short rows, 1.09 where all rows' last strips of 4096 columns came first
    calls = []
    for shape in ((16384, 4096), (4096, 16384)):
        x = torch.randn(shape, device="cuda")
        codes = torch.empty((shape[0], shape[1] // 2), dtype=torch.uint8, device="cuda")
        scales = torch.empty(fp4.fp4_scale_bytes(*shape), dtype=torch.uint8, device="cuda")
        calls.append((x, codes, scales, torch.empty(1, device="cuda")))
    times = [[], []]
    for _ in range(12):
        for call, t in zip(calls, times):
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            fp4.fp4_quantize(*call)
            e0.record()
            for _ in range(20):
                fp4.fp4_quantize(*call)
            e1.record()
            torch.cuda.synchronize()
            t.append(e0.elapsed_time(e1))
    assert np.median(times[1]) < 1.05 * np.median(times[0]), [np.median(t) for t in times]
