"""Parity of fp4_root_ns / fp4_root_ns_batched at the sizes and launch configurations the
benchmark and the scaling sweep run, and of the iterations after the first.

* square sweep sizes: the whole oracle at 4096 x 4096 (1 and 2 iterations); at 8192 and 16384 the
  first product on sampled 128 x 128 tiles, which the oracle computes from its own clip,
  normalisation and quantisation of the same input;
* the 28-matrix decoder-stack call exactly as the benchmark issues it (groups of 16 and of 8 + 4):
  bit-equality with single calls for matrices from the middle and the end of every group, and
  sampled oracle tiles on one of them;
* iteration 1, teacher-forced: the oracle runs one iteration from the GPU's own X1 (bit-identical
  inputs on both sides), every stage is compared as for iteration 0 - this reaches the G3 variant
  that reads X instead of the raw input and the second set of transposed operand copies;
* repeated calls give identical bytes (the epilogue warps hand buffers between the generic and
  the async proxy; a missing fence shows up as rare differing blocks).
"""
import numpy as np
import pytest
import torch

import oracle
import paper_2607_04422_b200 as fp4
from paper_2607_04422_b200 import workloads
from paper_2607_04422_b200.binding import (FP4_FLAG_FOUR_SIX, FP4_FLAG_KEEP_OPERANDS, FP4_FLAG_RHT,
                                           fp4_root_ns_workspace_layout)
from helpers import nibbles, sf_from_atoms

pytestmark = pytest.mark.gpu

TOL_OUT = 2e-3      # relative Frobenius error of the NS output per iteration count
TOL_STAGE = 1e-5    # stage outputs from bit-identical inputs: FP32 against FP64 accumulation
TOL_ORTH = 1e-2


def rel(a, b):
    a = a.astype(np.float64); b = b.astype(np.float64)
    return np.linalg.norm(a - b) / max(np.linalg.norm(b), 1e-300)


def orth_err(x):
    x = x.astype(np.float64)
    if x.shape[0] > x.shape[1]:
        x = x.T
    return np.linalg.norm(x @ x.T - np.eye(x.shape[0])) / np.sqrt(x.shape[0])


def run_gpu(G, steps, flags=0, seed=0):
    """G: device tensor.  Returns (out, workspace), both on the device."""
    m, n = G.shape
    out = torch.full((m, n), float("nan"), device="cuda")
    ws = torch.empty(fp4.fp4_root_ns_workspace_bytes(m, n, steps, flags), dtype=torch.uint8, device="cuda")
    fp4.fp4_root_ns(G, out, steps, fp4.NsParams.make(flags=flags, seed=seed), ws)
    assert fp4.fp4_last_device_status(ws) == 0
    return out, ws


class Workspace:
    """Reads single regions of a workspace without copying all of it to the host."""

    def __init__(self, ws, m, n, steps, flags):
        self.ws, self.lay = ws, fp4_root_ns_workspace_layout(m, n, steps, flags)
        self.s, self.l = min(m, n), max(m, n)
        self.sc = ws[self.lay.scalars:self.lay.scalars + 4096].cpu().numpy().view(np.float32)

    def f32_rows(self, off, cols, r0, r1):
        raw = self.ws[off + r0 * cols * 4:off + r1 * cols * 4].cpu().numpy()
        return raw.view(np.float32).reshape(r1 - r0, cols)

    def f32(self, off, rows, cols):
        return self.f32_rows(off, cols, 0, rows)

    def q(self, coff, soff, rows, cols):
        codes = self.ws[coff:coff + rows * cols // 2].cpu().numpy().reshape(rows, cols // 2)
        sf = sf_from_atoms(self.ws[soff:soff + rows * cols // 16].cpu().numpy(), rows, cols // 16)
        return codes, sf


def check_sampled_tiles_of_A(G_np, G_dev, tiles=6, seed=0):
    """Iteration 0's A = qX qX^T on sampled 128 x 128 tiles of the upper triangle, against the
    oracle's product of its own quantisation of its own X0 (work orientation s x l)."""
    m, n = G_np.shape
    flags = FP4_FLAG_KEEP_OPERANDS
    _, ws = run_gpu(G_dev, 1, flags)
    w = Workspace(ws, m, n, 1, flags)
    X0 = oracle.root_ns(G_np, steps=0)
    if m > n:
        X0 = np.ascontiguousarray(X0.T)
    qx = oracle.quantize(X0)
    assert w.sc[w.lay.idx_sg_X0] == np.float32(qx[2])
    rng = np.random.default_rng(seed)
    s = w.s
    for _ in range(tiles):
        i = int(rng.integers(0, s // 128)); j = int(rng.integers(i, s // 128))
        rows = slice(128 * i, 128 * i + 128); cols = slice(128 * j, 128 * j + 128)
        want = oracle.gemm_nt_q((qx[0][rows], qx[1][rows], qx[2]), (qx[0][cols], qx[1][cols], qx[2]))
        got = w.f32_rows(w.lay.A, s, 128 * i, 128 * i + 128)[:, cols]
        assert np.abs(got - want).max() <= TOL_STAGE * np.abs(want).max(), (i, j)


# ------------------------------------------------------------------------------------------
# the scaling sweep (square Gaussian inputs, seed 1)
def test_sweep_4096_whole_oracle_one_and_two_iterations():
    G = workloads.gaussian(4096, 4096, seed=1)
    Gd = torch.from_numpy(G).cuda()
    want2, tr = oracle.root_ns(G, steps=2, trace_iter=0)       # X after iteration 0 = the 1-iteration result
    got1, _ = run_gpu(Gd, 1)
    got2, _ = run_gpu(Gd, 2)
    for got, want in ((got1.cpu().numpy(), tr["X_out"]), (got2.cpu().numpy(), want2)):
        assert rel(got, want) <= TOL_OUT, rel(got, want)
        assert abs(orth_err(got) - orth_err(want)) <= TOL_ORTH


@pytest.mark.parametrize("size", [8192, 16384])
def test_sweep_large_sizes_sampled_tiles(size):
    G = workloads.gaussian(size, size, seed=1)
    Gd = torch.from_numpy(G).cuda()
    check_sampled_tiles_of_A(G, Gd, tiles=6, seed=size)
    del Gd
    torch.cuda.empty_cache()


# ------------------------------------------------------------------------------------------
# the benchmark's call: 28 matrices, default grouping
def test_decoder_stack_call_as_benchmarked():
    specs = workloads.stack_3b_shapes(4)
    mats = [workloads.gradient_like(m, n, seed=seed) for _, m, n, seed in specs]
    Gs = [torch.from_numpy(g).cuda() for g in mats]
    outs = [torch.empty_like(g) for g in Gs]
    shapes = [tuple(g.shape) for g in Gs]
    ws = torch.empty(fp4.fp4_root_ns_batched_workspace_bytes(shapes, 5), dtype=torch.uint8, device="cuda")
    fp4.fp4_root_ns_batched(Gs, outs, 5, None, ws)
    assert fp4.fp4_last_device_status(ws) == 0
    # groups in call order: the sixteen 3072 x 3072; the eight wide and four tall 3072 x 8192 / 8192 x 3072
    square = [i for i, sh in enumerate(shapes) if sh == (3072, 3072)]
    rect = [i for i, sh in enumerate(shapes) if sh != (3072, 3072)]
    assert len(square) == 16 and len(rect) == 12
    picks = [square[7], square[8], square[15], rect[5], rect[6], rect[10], rect[11]]
    assert {shapes[i] for i in picks} == {(3072, 3072), (3072, 8192), (8192, 3072)}
    for i in picks:
        single, _ = run_gpu(Gs[i], 5)
        assert torch.equal(outs[i], single), (i, shapes[i])
        assert bool(torch.isfinite(single).all())
    # the same call again on the same workspace, other outputs: nothing stale is picked up
    outs2 = [torch.full_like(g, float("nan")) for g in Gs]
    fp4.fp4_root_ns_batched(Gs, outs2, 5, None, ws)
    assert fp4.fp4_last_device_status(ws) == 0
    for a, b in zip(outs, outs2):
        assert torch.equal(a, b)
    del outs, outs2, ws
    torch.cuda.empty_cache()
    # oracle tiles for one tall matrix of the last group (work orientation: its transpose)
    i = rect[11]
    assert shapes[i] == (8192, 3072)
    check_sampled_tiles_of_A(mats[i], Gs[i], tiles=4, seed=3)


def test_batched_twice_on_one_workspace_with_other_shapes():
    """A workspace is reused by a second batched call with different matrices and shapes: the
    second result equals single calls (descriptors of the first call must not survive anywhere)."""
    first = [(512, 1024, 1), (512, 512, 2), (1024, 512, 3)]
    second = [(256, 512, 4), (768, 768, 5), (512, 256, 6), (256, 512, 7)]
    shapes1 = [(m, n) for m, n, _ in first]; shapes2 = [(m, n) for m, n, _ in second]
    need = max(fp4.fp4_root_ns_batched_workspace_bytes(shapes1, 3), fp4.fp4_root_ns_batched_workspace_bytes(shapes2, 3))
    ws = torch.empty(need, dtype=torch.uint8, device="cuda")
    for specs in (first, second):
        mats = [torch.from_numpy(workloads.gradient_like(m, n, seed=sd)).cuda() for m, n, sd in specs]
        outs = [torch.empty_like(g) for g in mats]
        fp4.fp4_root_ns_batched(mats, outs, 3, None, ws)
        assert fp4.fp4_last_device_status(ws) == 0
    for g, o in zip(mats, outs):
        single, _ = run_gpu(g, 3)
        assert torch.equal(o, single)


# ------------------------------------------------------------------------------------------
# iteration 1, teacher-forced from the GPU's own X1
QMODES = {"base": (False, False), "paper": (True, True)}


@pytest.mark.parametrize("qmode", ["base", "paper"])
@pytest.mark.parametrize("shape", [(256, 512), (512, 256), (384, 384), (512, 1024)])
def test_iteration_one_every_stage_teacher_forced(shape, qmode):
    m, n = shape
    rht, fs = QMODES[qmode]
    seed = 31
    flags = FP4_FLAG_KEEP_OPERANDS | (FP4_FLAG_RHT if rht else 0) | (FP4_FLAG_FOUR_SIX if fs else 0)
    G = torch.from_numpy(workloads.gradient_like(m, n, seed=11)).cuda()
    out1, ws1 = run_gpu(G, 1, flags, seed)
    out2, ws2 = run_gpu(G, 2, flags, seed)
    w1 = Workspace(ws1, m, n, 1, flags); w2 = Workspace(ws2, m, n, 2, flags)
    s, l, lay = w1.s, w1.l, w1.lay
    X1 = out1.cpu().numpy(); X2 = out2.cpu().numpy()
    if m > n:
        X1 = np.ascontiguousarray(X1.T); X2 = np.ascontiguousarray(X2.T)
    amax1, sg1 = w1.sc[lay.idx_amax_X0 + 1], w1.sc[lay.idx_sg_X0 + 1]
    assert amax1 == np.abs(X1).max()
    assert w2.sc[lay.idx_amax_X0 + 1] == amax1 and w2.sc[lay.idx_sg_X0 + 1] == sg1     # the 2-step run passed through X1
    want, amax2, sg2, tr = oracle.ns_iteration(X1, 1, float(amax1), float(sg1), last=True, rht=rht, four_six=fs, seed=seed)
    # G1 of iteration 1
    A = w2.f32(lay.A, s, s)
    mask = np.kron(np.triu(np.ones((s // 128, s // 128))), np.ones((128, 128))).astype(bool)
    assert np.abs(A[mask] - tr["A"][mask]).max() <= TOL_STAGE * np.abs(tr["A"]).max()
    assert w2.sc[lay.idx_sg_A0 + 1] == np.float32(tr["sg_A"])
    assert abs(w2.sc[lay.idx_amax_A0 + 1] - np.abs(tr["A"]).max()) <= 1e-6 * np.abs(tr["A"]).max()
    # qA, qB of iteration 1 (both triangles)
    for name, co, so in (("qA", lay.qA_codes, lay.qA_scales), ("qB", lay.qB_codes, lay.qB_scales)):
        codes, sf = w2.q(co, so, s, s)
        sf_diff = sf != tr[name + "_scales"]
        assert sf_diff.mean() < (6e-3 if fs else 2e-3), (name, sf_diff.mean())
        g, w = nibbles(codes), nibbles(tr[name + "_codes"])
        bad = (g != w) & ~np.repeat(sf_diff, 16, axis=1)
        assert bad.mean() < 2e-3, (name, bad.mean())
        if bad.any():
            assert np.abs((g[bad] & 7).astype(int) - (w[bad] & 7).astype(int)).max() <= 1, name
    assert w2.sc[lay.idx_sg_B0 + 1] == np.float32(tr["sg_B"])
    # G3 of iteration 1: X2, and the operand copies written for iteration 2 (the other set of X^T copies)
    assert rel(X2, want) < 2e-4
    assert w2.sc[lay.idx_amax_X0 + 2] == np.abs(X2).max()
    assert w2.sc[lay.idx_sg_X0 + 2] == np.float32(sg2)
    qopt = dict(rht=rht, mask=oracle.rht_mask(seed, 4) if rht else 0, four_six=fs)
    oc, os_, _ = oracle.quantize(X2, s_g=float(sg2), **qopt)
    codes, sf = w2.q(lay.qX_codes, lay.qX_scales, s, l)
    assert np.array_equal(codes, oc) and np.array_equal(sf, os_)
    oc, os_, _ = oracle.quantize(np.ascontiguousarray(X2.T), s_g=float(sg2), **qopt)
    codes, sf = w2.q(lay.qXt_codes[0], lay.qXt_scales[0], l, s)
    assert np.array_equal(codes, oc) and np.array_equal(sf, os_)


# ------------------------------------------------------------------------------------------
def test_repeated_calls_give_identical_bytes():
    """Every quantised output and the result of 60 identical calls, on a shape large enough for
    several tiles per CTA pair; the workspace starts from a poison pattern each time."""
    m = n = 2048
    flags = FP4_FLAG_KEEP_OPERANDS
    G = torch.from_numpy(workloads.gradient_like(m, n, seed=17)).cuda()
    lay = fp4_root_ns_workspace_layout(m, n, 2, flags)
    nbytes = fp4.fp4_root_ns_workspace_bytes(m, n, 2, flags)
    regions = [(lay.scalars, 4096), (lay.qX_codes, m * n // 2), (lay.qX_scales, m * n // 16),
               (lay.qXt_codes[0], m * n // 2), (lay.qXt_scales[0], m * n // 16),
               (lay.qA_codes, m * m // 2), (lay.qA_scales, m * m // 16), (lay.qB_codes, m * m // 2), (lay.qB_scales, m * m // 16)]
    ref = None
    for r in range(60):
        ws = torch.full((nbytes,), 0xFF, dtype=torch.uint8, device="cuda")
        out = torch.empty_like(G)
        fp4.fp4_root_ns(G, out, 2, fp4.NsParams.make(flags=flags), ws)
        cur = [out] + [ws[o:o + sz].clone() for o, sz in regions]
        assert fp4.fp4_last_device_status(ws) == 0
        if ref is None:
            ref = cur
            continue
        for k, (a, b) in enumerate(zip(cur, ref)):
            assert torch.equal(a, b), (r, k)


# ------------------------------------------------------------------------------------------
# long contractions: G2 / G3 with four operand stages and one chunk buffer per warp (K >= 4096, with the quantiser options
# 5120), tiles in bands of eight rows (column operands of 32 MB and more)
@pytest.mark.parametrize("m,n,qmode", [(4224, 16000, "base"), (5248, 5248, "paper"), (16000, 4224, "base")])
def test_long_contractions_sampled_tiles(m, n, qmode):
    """Odd numbers of 128-blocks both ways, the last band one row high.  The products are recomputed from the GPU's own
    operands, so the bound is that of a stage: FP32 against FP64 accumulation."""
    rht, fs = QMODES[qmode]
    flags = FP4_FLAG_KEEP_OPERANDS | (FP4_FLAG_RHT if rht else 0) | (FP4_FLAG_FOUR_SIX if fs else 0)
    G = workloads.gradient_like(m, n, seed=3)
    abc = (3.4445, -4.775, 2.0315)
    Gd = torch.from_numpy(G).cuda()
    out = torch.full((m, n), float("nan"), device="cuda")
    ws = torch.empty(fp4.fp4_root_ns_workspace_bytes(m, n, 1, flags), dtype=torch.uint8, device="cuda")
    fp4.fp4_root_ns(Gd, out, 1, fp4.NsParams.make(abc=abc, flags=flags, seed=9), ws)
    assert fp4.fp4_last_device_status(ws) == 0
    w = Workspace(ws, m, n, 1, flags)
    s, l, lay, sc = w.s, w.l, w.lay, w.sc
    a, b, c = (np.float32(x) for x in abc)
    tau, inv = sc[lay.idx_tau], sc[lay.idx_inv]
    work, res = (G, out) if m <= n else (G.T, out.T)
    qB, qXt, qA = w.q(lay.qB_codes, lay.qB_scales, s, s), w.q(lay.qXt_codes[0], lay.qXt_scales[0], l, s), \
        w.q(lay.qA_codes, lay.qA_scales, s, s)
    sgA, sgB, sgX = sc[lay.idx_sg_A0], sc[lay.idx_sg_B0], sc[lay.idx_sg_X0]
    nb, nl = s // 128, l // 128
    rng = np.random.default_rng(0)
    pick = [(0, 0), (nb - 1, nl - 1), (nb - 1, 0), (7, nl - 1), (8, 1)] + [(int(rng.integers(nb)), int(rng.integers(nl))) for _ in range(8)]
    for i, j in pick:
        r, q = slice(128 * i, 128 * i + 128), slice(128 * j, 128 * j + 128)
        P = oracle.gemm_nt_q((qB[0][r], qB[1][r], sgB), (qXt[0][q], qXt[1][q], sgX))
        want = a * (np.clip(work[r, q], -tau, tau) * inv) + P
        got = res[r, q].cpu().numpy()
        assert np.abs(got - want).max() <= TOL_STAGE * np.abs(want).max(), (i, j)
        if qmode == "base":
            k = max(i, j % nb); i2 = min(i, j % nb)
            r, q = slice(128 * i2, 128 * i2 + 128), slice(128 * k, 128 * k + 128)
            S = oracle.gemm_nt_q((qA[0][r], qA[1][r], sgA), (qA[0][q], qA[1][q], sgA))
            B = b * w.f32_rows(lay.A, s, 128 * i2, 128 * i2 + 128)[:, q] + c * S
            for tile, rr, qq in ((B, r, q), (np.ascontiguousarray(B.T), q, r)):
                oc, osf, _ = oracle.quantize(tile, s_g=float(sgB))
                cols = slice(qq.start // 2, qq.stop // 2); blocks = slice(qq.start // 16, qq.stop // 16)
                sf_bad = osf != qB[1][rr, blocks]
                # the two accumulations differ in the last places, so a value on a rounding boundary may fall either way
                assert sf_bad.mean() < 5e-3 and (nibbles(oc) != nibbles(qB[0][rr, cols]))[~np.repeat(sf_bad, 16, axis=1)].mean() < 2e-3


def test_long_contraction_bf16_storage_whole_oracle():
    G = workloads.gradient_like(4224, 4352, seed=5)
    got, _ = run_gpu(torch.from_numpy(G).cuda(), 2, fp4.FP4_FLAG_STORE_BF16)
    want = oracle.root_ns(G, steps=2, store_bf16=True)
    got = got.cpu().numpy()
    assert rel(got, want) <= TOL_OUT and abs(orth_err(got) - orth_err(want)) <= TOL_ORTH
