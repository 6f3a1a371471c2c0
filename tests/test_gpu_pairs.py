"""Tensor-core kernel on block pairs (cta_group::2: tiles of 256 weight rows over clusters of two blocks): both tile widths,
odd numbers of 128-row tiles, token counts at the edges of boxes and halves of boxes, whole, split and half tiles, many
tiles per pair, and every epilogue."""
import numpy as np
import pytest
import torch

import oracle
from helpers import check_output, dev_weight, dev_x
from test_gpu_prefill import B, run_ex, run_rope  # noqa: F401  (B: fixture)
from paper_2512_03383_b200 import synth

pytestmark = pytest.mark.gpu

TOL = 5e-4       # as the other tests of this kernel: weights rounded once to fp16, fp32 sums


@pytest.fixture(autouse=True)
def _reset(B):
    B.set_path(B.PATH_PREFILL)
    yield
    B.set_path(B.PATH_AUTO)
    B.reset_options()


@pytest.mark.parametrize("width", [1, 2])
@pytest.mark.parametrize("M", [129, 256, 300, 385, 513, 1100])
@pytest.mark.parametrize("dtype", ["f16", "bf16"])
def test_whole_tiles(B, M, dtype, width):
    B.set_option("prefill_streamk", 0)
    rng = np.random.default_rng(2000 + M)
    qw = synth.draw_qweight(rng, 700, 1024)
    dw = dev_weight(qw)
    bias = synth.to_dtype_values(rng.standard_normal(700).astype(np.float32), dtype)
    for (k_in, k_out) in ((1024, 700), (652, 132)):
        x = synth.draw_x(rng, M, k_in, dtype)
        got = []
        for pair in (width, 0):
            B.set_option("prefill_pair", pair)
            y, ref = run_ex(B, qw, dw, x, dtype, None, k_in, None, k_out, bias=bias, ldx_pad=8 - k_in % 8 if k_in % 8 else 0, ldy_pad=3)
            got.append(y.clone())
        check_output(got[0], ref, dtype, TOL, "pairs M=%d %s k=(%d,%d)" % (M, dtype, k_in, k_out))
        assert torch.equal(got[0], got[1]), "a tile's k-blocks are summed in the same order by one block and by a pair"
    assert B.workspace_status() == 0


@pytest.mark.parametrize("width", [1, 2])
@pytest.mark.parametrize("grid", [1, 2, 3, 7])
@pytest.mark.parametrize("form", [0, 1, 2])
def test_split_tiles_and_many_tiles_per_pair(B, grid, form, width):
    B.set_option("prefill_pair", width)
    B.set_option("prefill_grid", grid)
    B.set_option("prefill_streamk", form)
    rng = np.random.default_rng(2100 + grid)
    for (N, K, M) in ((900, 256, 600), (300, 1024, 300), (1500, 128, 1100)):
        qw = synth.draw_qweight(rng, N, K)
        dw = dev_weight(qw)
        x = synth.draw_x(rng, M, K, "f16")
        y, ref = run_ex(B, qw, dw, x, "f16", None, K, None, N)
        check_output(y, ref, "f16", TOL, "N=%d K=%d M=%d grid %d form %d" % (N, K, M, grid, form))
        if form < 2:
            y2, _ = run_ex(B, qw, dw, x, "f16", None, K, None, N)
            assert torch.equal(y, y2)
    for (g, r) in run_rope(B, rng, 300, 512, 6, 2, 128, 84, 5e5, "f16", bias=True):
        check_output(g, r, "f16", TOL, "rope grid %d form %d" % (grid, form))
    im = synth.map_per_head(8, 128, 104)
    qw = synth.draw_qweight(rng, 200, 1024)
    x = synth.draw_x(rng, 300, synth.map_size(im), "bf16")
    y, ref = run_ex(B, qw, dev_weight(qw), x, "bf16", im, 0, None, 200, ldx_pad=8)
    check_output(y, ref, "bf16", TOL, "per-head input map")
    assert B.workspace_status() == 0


@pytest.mark.parametrize("width", [1, 2])
def test_half_tiles_and_gated_product(B, width):
    """Half tiles: three tiles of 512 tokens on two pairs; the gated pair job and the down projection behind it."""
    B.set_option("prefill_pair", width)
    B.set_option("prefill_dual", 3)
    B.set_option("prefill_grid", 2)
    rng = np.random.default_rng(2200)
    qw = synth.draw_qweight(rng, 700, 512)
    x = synth.draw_x(rng, 500, 512, "f16")
    y, ref = run_ex(B, qw, dev_weight(qw), x, "f16", None, 512, None, 700)
    check_output(y, ref, "f16", TOL, "half tiles")
    B.reset_options()
    B.set_option("prefill_pair", width)
    hidden, inter, k_int, M = 512, 1024, 872, 300
    ws = [synth.draw_qweight(rng, n, k) for n, k in ((inter, hidden), (inter, hidden), (hidden, inter))]
    ds = [dev_weight(w) for w in ws]
    x = synth.draw_x(rng, M, hidden, "f16")
    h = torch.zeros((M, k_int), dtype=torch.float16, device="cuda")
    y = torch.zeros((M, hidden), dtype=torch.float16, device="cuda")
    B.mlp_swiglu(dev_x(x, "f16"), hidden, *ds[0][1:], *ds[1][1:], *ds[2][1:], M, hidden, inter, k_int, h, k_int, y, hidden)
    torch.cuda.synchronize()
    a = []
    for w, d in zip(ws, ds):
        a += [d[0], w.scales, w.zeros]
    h_ref, y_ref = oracle.mlp_swiglu(x, *a, k_int, h_dtype="f16")
    check_output(h, h_ref, "f16", TOL, "h")
    check_output(y, y_ref, "f16", 1e-3, "y")
    assert B.workspace_status() == 0


@pytest.mark.parametrize("share", [2, 3, 4])
@pytest.mark.parametrize("M", [129, 256, 300])
@pytest.mark.parametrize("dtype", ["f16", "bf16"])
def test_tiles_shared_by_the_pairs_of_a_cluster(B, M, dtype, share):
    """A part of the contraction per pair, sums exchanged inside the cluster: k-block counts that do not divide, ragged
    rows and tokens, every epilogue, the same bits on every run."""
    B.set_option("prefill_pair", 1)
    B.set_option("prefill_streamk", 10 + share)
    rng = np.random.default_rng(2300 + M)
    qw = synth.draw_qweight(rng, 700, 1024)
    dw = dev_weight(qw)
    bias = synth.to_dtype_values(rng.standard_normal(700).astype(np.float32), dtype)
    for (k_in, k_out) in ((1024, 700), (652, 132)):
        x = synth.draw_x(rng, M, k_in, dtype)
        y, ref = run_ex(B, qw, dw, x, dtype, None, k_in, None, k_out, bias=bias, ldx_pad=8 - k_in % 8 if k_in % 8 else 0, ldy_pad=3)
        check_output(y, ref, dtype, TOL, "shared by %d M=%d %s k=(%d,%d)" % (share, M, dtype, k_in, k_out))
        y2, _ = run_ex(B, qw, dw, x, dtype, None, k_in, None, k_out, bias=bias, ldx_pad=8 - k_in % 8 if k_in % 8 else 0, ldy_pad=3)
        assert torch.equal(y, y2)
    for helpers in (1, 0):
        B.set_option("prefill_helpers", helpers)
        for (g, r) in run_rope(B, rng, M, 512, 6, 2, 128, 84, 5e5, dtype, bias=True):
            check_output(g, r, dtype, TOL, "rope shared by %d" % share)
        im = synth.map_per_head(8, 128, 104)
        x = synth.draw_x(rng, M, synth.map_size(im), dtype)
        y, ref = run_ex(B, qw, dw, x, dtype, im, 0, None, 200, ldx_pad=8)
        check_output(y, ref, dtype, TOL, "per-head input map shared by %d" % share)
    assert B.workspace_status() == 0


@pytest.mark.parametrize("dtype", ["f16", "bf16"])
@pytest.mark.parametrize("M,N,K", [(300, 700, 512), (200, 300, 1024), (1100, 1500, 128), (48, 300, 2048), (12, 300, 2048), (100, 300, 1920)])
def test_refused_cluster_launches(B, M, N, K, dtype):
    """A device that does not take the clusters a plan asks for: the call runs on single blocks instead of failing (pairs of
    one and two boxes, pairs that share a tile, the batch kernel's shared tiles, tiles shared by two blocks)."""
    rng = np.random.default_rng(2350 + M)
    qw = synth.draw_qweight(rng, N, K)
    dw = dev_weight(qw)
    x = synth.draw_x(rng, M, K, dtype)
    B.set_option("prefill_pair", 3)
    for split in (-1, 3, 12):
        B.set_option("prefill_streamk", split)
        y, ref = run_ex(B, qw, dw, x, dtype, None, K, None, N)
        check_output(y, ref, dtype, TOL, "refused clusters M=%d %s split %d" % (M, dtype, split))
    assert B.workspace_status() == 0
