"""Batch kernel (17 to 128 rows): contractions long enough that its rings wrap many times, alone and back to back."""
import numpy as np
import pytest
import torch

import oracle
from helpers import check_output, dev_weight, dev_x
from test_gpu_prefill import B, run_ex  # noqa: F401  (B: fixture)
from paper_2512_03383_b200 import synth

pytestmark = pytest.mark.gpu

TOL = 5e-4       # as the other tensor-core tests: weights rounded once to fp16, fp32 sums


def in_flight(B, dw, x, dtype, in_map, k_in, N, K, count):
    """`count` launches behind one another with nothing between them, each into an output of its own: blocks of two launches
    share the SMs and their tensor memory, codes are fetched before the launch in front is complete, and every launch uses
    the slots of the one in front."""
    xd = dev_x(x, dtype)
    out = [torch.full((x.shape[0], N), -77.0, device="cuda", dtype=xd.dtype) for _ in range(count)]
    for y in out:
        B.qlinear_ex(xd, xd.shape[1], *dw[1:], None, x.shape[0], K, N, in_map, k_in, None, N, y, N)
    torch.cuda.synchronize()
    return out


@pytest.mark.parametrize("M", [17, 48, 64, 100, 128])
@pytest.mark.parametrize("split", [0, -1])
def test_long_contractions(B, M, split):
    B.set_path(B.PATH_PREFILL)
    B.set_option("prefill_streamk", split)
    rng = np.random.default_rng(2400 + M)
    for (N, K) in ((640, 8192), (1500, 4096)):
        qw = synth.random_qweight_fast(rng, N, K)
        dw = dev_weight(qw)
        x = synth.draw_x(rng, M, K, "f16")
        y, ref = run_ex(B, qw, dw, x, "f16", None, K, None, N)
        check_output(y, ref, "f16", TOL, "M=%d N=%d K=%d" % (M, N, K))
        for again in in_flight(B, dw, x, "f16", None, K, N, K, 20):
            assert torch.equal(again, y)
    assert B.workspace_status() == 0
    B.set_path(B.PATH_AUTO)
    B.reset_options()


@pytest.mark.parametrize("M", [1, 12, 15, 16])
@pytest.mark.parametrize("N,K,take", [(8, 256, 256), (136, 1024, 1000), (640, 8192, 8192), (1500, 4096, 3976), (200, 1024, "72"),
                                      (200, 1024, "104"), (328, 2048, "96"), (130, 1024, "128")])
@pytest.mark.parametrize("split", [0, -1])
def test_exact_codes(B, M, N, K, take, split):
    """Up to 16 fp16 rows; `take`: leading channels, or the kept channels of heads of 128.  Codes and activations enter
    unrounded, so beyond the output's rounding only fp32 sums remain: 8 + K / 128 <= 72 of them in a chain, 2^-23 each of
    sum |terms|, which is up to 25 times the largest output: 2.2e-4."""
    B.set_path(B.PATH_PREFILL)
    B.set_option("prefill_streamk", split)
    rng = np.random.default_rng(7 * M + N + K)
    qw = synth.random_qweight_fast(rng, N, K)
    dw = dev_weight(qw)
    im = synth.map_per_head(K // 128, 128, int(take)) if isinstance(take, str) else None
    k_in = 0 if im else take
    x = synth.draw_x(rng, M, synth.map_size(im) if im else k_in, "f16")
    y, ref = run_ex(B, qw, dw, x, "f16", im, k_in, None, N)
    check_output(y, ref, "f16", 3e-4, "M=%d N=%d K=%d %s" % (M, N, K, take))
    for again in in_flight(B, dw, x, "f16", im, k_in, N, K, 20):
        assert torch.equal(again, y)
    assert B.workspace_status() == 0
    B.set_path(B.PATH_AUTO)
    B.reset_options()


@pytest.mark.parametrize("M,dtype", [(12, "f16"), (12, "bf16"), (40, "f16"), (40, "bf16"), (128, "f16"), (128, "bf16")])
@pytest.mark.parametrize("heads", [False, True])
def test_code_ring_wraps_in_every_instance(B, M, dtype, heads):
    """A whole contraction per block (32 stages in rings of two to six), plain and per-head, both types, codes multiplied as
    they are and rounded to fp16: a slot handed back before its codes were read shows as wrong rows."""
    B.set_path(B.PATH_PREFILL)
    B.set_option("prefill_streamk", 0)
    rng = np.random.default_rng(2500 + M)
    N, K = 700, 8192
    qw = synth.random_qweight_fast(rng, N, K)
    dw = dev_weight(qw)
    im = synth.map_per_head(K // 128, 128, 104) if heads else None
    x = synth.draw_x(rng, M, synth.map_size(im) if im else K, dtype)
    y, ref = run_ex(B, qw, dw, x, dtype, im, 0 if im else K, None, N)
    check_output(y, ref, dtype, TOL, "M=%d %s heads %d" % (M, dtype, heads))
    for again in in_flight(B, dw, x, dtype, im, 0 if im else K, N, K, 20):
        assert torch.equal(again, y)
    assert B.workspace_status() == 0
    B.set_path(B.PATH_AUTO)
    B.reset_options()


@pytest.mark.parametrize("option,value", [("decode_kp", 2), ("decode_rp", 20), ("decode_stages", 2), ("decode_xstream", 1),
                                          ("decode_split_batch", 1), ("decode_i8", 0)])
def test_options_of_the_decode_kernel_ask_for_it(B, option, value):
    """The automatic choice at twelve to sixteen rows is the batch kernel, unless an option of the decode kernel is set: then
    the bits are those of the decode kernel."""
    rng = np.random.default_rng(2600)
    qw = synth.random_qweight_fast(rng, 300, 2048)
    dw = dev_weight(qw)
    x = synth.draw_x(rng, 16, 2048, "f16")
    B.set_option(option, value)
    got = []
    for path in (B.PATH_AUTO, B.PATH_DECODE):
        B.set_path(path)
        y, ref = run_ex(B, qw, dw, x, "f16", None, 2048, None, 300)
        check_output(y, ref, "f16", TOL, "%s=%d path %d" % (option, value, path))
        got.append(y.clone())
    B.reset_options()
    B.set_path(B.PATH_AUTO)
    batch, _ = run_ex(B, qw, dw, x, "f16", None, 2048, None, 300)
    assert torch.equal(got[0], got[1]) and not torch.equal(got[0], batch)


@pytest.mark.parametrize("M,dtype", [(12, "f16"), (16, "f16"), (12, "bf16"), (40, "f16"), (128, "f16"), (128, "bf16")])
@pytest.mark.parametrize("split", [0, -1])
def test_chain_of_dependent_launches(B, M, dtype, split):
    """Every launch reads what the one in front wrote, and its matrix has another shape, so that the number of blocks that
    share a tile changes from launch to launch: the bits are those without programmatic dependent launch."""
    B.set_path(B.PATH_PREFILL)
    B.set_option("prefill_streamk", split)
    rng = np.random.default_rng(2700 + M)
    sizes = [(1536, 512), (4096, 1536), (512, 4096)]               # (N, K), in turn
    ws = [synth.draw_qweight(rng, n, k) for n, k in sizes]
    ds = [dev_weight(w) for w in ws]
    x = synth.draw_x(rng, M, 512, dtype) * np.float32(2.0 ** -6)
    xd = torch.from_numpy(x).cuda().to(torch.float16 if dtype == "f16" else torch.bfloat16)

    def chain(pdl):
        B.set_option("pdl", pdl)
        outs, src = [], xd
        for i in range(9):
            (n, k), d = sizes[i % 3], ds[i % 3]
            y = torch.zeros((M, n), dtype=xd.dtype, device="cuda")
            B.qlinear_ex(src, k, *d[1:], None, M, k, n, None, k, None, n, y, n)
            outs.append(y)
            src = y
            if i % 3 == 2:                                         # (kept in range, on the same stream)
                src = y * (2.0 ** -6 / y.abs().amax().clamp_min(1e-3)).to(y.dtype)
        torch.cuda.synchronize()
        return outs

    off = chain(0)
    assert all(torch.isfinite(y.float()).all() and y.abs().amax() > 0 for y in off)
    for rep in range(5):
        for i, (a, b) in enumerate(zip(chain(1), off)):
            assert torch.equal(a, b), "link %d repeat %d" % (i, rep)
    ref = oracle.qlinear(xd.float().cpu().numpy(), ds[0][0], ws[0].scales, ws[0].zeros, oracle.leading(1536), oracle.leading(512))
    check_output(off[0], ref, dtype, TOL, "first link M=%d %s" % (M, dtype))
    assert B.workspace_status() == 0
    B.set_path(B.PATH_AUTO)
    B.reset_options()


@pytest.mark.parametrize("M", [17, 40, 64, 128])
@pytest.mark.parametrize("heads,dim,keep", [(8, 128, 108), (10, 128, 84), (6, 128, 68), (4, 128, 124), (16, 64, 52), (12, 64, 12), (20, 64, 60)])
def test_heads_that_keep_4_mod_8_channels(B, M, heads, dim, keep):
    """Every second head's activations begin 4 channels behind a 16-byte boundary and are read in place; whole and shared
    tiles, a row pitch with a gap, ragged rows.  Tolerance as for the other maps of this kernel."""
    rng = np.random.default_rng(31 * M + keep)
    im = synth.map_per_head(heads, dim, keep)
    qw = synth.draw_qweight(rng, 300, heads * dim)
    dw = dev_weight(qw)
    x = synth.draw_x(rng, M, synth.map_size(im), "f16")
    for split in (0, -1):
        B.set_option("prefill_streamk", split)
        y, ref = run_ex(B, qw, dw, x, "f16", im, 0, None, 300, ldx_pad=8 + (-x.shape[1]) % 8, ldy_pad=1)
        check_output(y, ref, "f16", TOL, "M=%d %d heads of %d keep %d" % (M, heads, dim, keep))
    assert B.workspace_status() == 0
    B.reset_options()


@pytest.mark.parametrize("M", [17, 64, 128])
@pytest.mark.parametrize("fam", [(256, 128, 108, 6), (512, 128, 84, 3), (256, 64, 52, 9), (256, 64, 60, 12)])
def test_heads_that_keep_4_mod_8_channels_behind_channel_0(B, M, fam):
    """The same with the first head on a later 256-channel boundary, the only one where they are read in place."""
    rng = np.random.default_rng(37 * M + fam[2])
    qw = synth.draw_qweight(rng, 200, 1024)
    dw = dev_weight(qw)
    x = synth.draw_x(rng, M, fam[2] * fam[3], "f16")
    for split in (0, -1):
        B.set_option("prefill_streamk", split)
        y, ref = run_ex(B, qw, dw, x, "f16", [fam], 0, None, 200, ldx_pad=8 + (-x.shape[1]) % 8, ldy_pad=1)
        check_output(y, ref, "f16", TOL, "M=%d %s" % (M, fam))
    assert B.workspace_status() == 0
    B.reset_options()
