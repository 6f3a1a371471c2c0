"""A caller workspace of exactly the advertised size is enough and nothing is written behind it: the workspace
sits in front of a band of canary bytes that must survive every kind of launch (split input channels, streamed
activations of 5..16 rows, re-laid activations, tiles split along K on the tensor cores, the fp16 copy of bf16
activations, the SwiGLU block)."""
import numpy as np
import pytest
import torch

import oracle
from helpers import check_output, dev_weight, dev_x
from paper_2512_03383_b200 import synth
from test_gpu_parity import run_ex
from test_gpu_mlp import draw_mlp, run_mlp, TOL_H, TOL_Y

pytestmark = pytest.mark.gpu
BAND = 1 << 20
CANARY = 0xA5


@pytest.fixture(scope="module")
def B():
    from paper_2512_03383_b200 import binding
    return binding


@pytest.fixture(autouse=True)
def _reset(B):
    yield
    B.set_path(B.PATH_AUTO)
    B.reset_options()


def guarded(B, nbytes):
    buf = torch.full((nbytes + BAND,), CANARY, dtype=torch.uint8, device="cuda")
    ws = buf[:nbytes]
    B.workspace_init(ws)
    return buf, ws


def band_intact(buf, nbytes):
    torch.cuda.synchronize()
    return bool((buf[nbytes:] == CANARY).all())


@pytest.mark.parametrize("M", [1, 4, 7, 8, 9, 16, 40, 300, 700])
def test_linear_layers_stay_inside_the_advertised_workspace(B, M):
    rng = np.random.default_rng(1200 + M)
    dtype = "f16"
    for (N, K, k_in, k_out) in [(200, 2304, 2304, 200), (70, 8192, 8192, 70), (330, 1024, 1020, 330), (1100, 512, 512, 1100)]:
        qw = synth.draw_qweight(rng, N, K)
        dw = dev_weight(qw)
        nbytes = B.workspace_bytes(M, K, N)
        buf, ws = guarded(B, nbytes)
        x = synth.draw_x(rng, M, k_in, dtype)
        for opts in ({}, {"decode_kp": 3, "decode_rp": 5}, {"decode_xstream": 1}, {"prefill_streamk": 1, "prefill_grid": 5},
                     {"prefill_streamk": 1, "prefill_grid": 5, "prefill_dual": 1}):
            B.reset_options()
            for k, v in opts.items():
                B.set_option(k, v)
            y, ref = run_ex(B, qw, dw, x, dtype, None, k_in, None, k_out, ldy_pad=3, workspace=ws)
            check_output(y, ref, dtype, 5e-4, "M=%d %s %s" % (M, (N, K, k_in, k_out), opts))
            assert band_intact(buf, nbytes), "wrote behind the workspace: M=%d %s %s" % (M, (N, K), opts)
            assert B.workspace_status(ws) == 0
    # per-head input maps with keep counts off the 8-channel grid: the activations are re-laid inside the workspace
    qw = synth.draw_qweight(rng, 256, 1024)
    dw = dev_weight(qw)
    im = synth.map_per_head(8, 128, 108)
    nbytes = B.workspace_bytes(M, 1024, 256)
    buf, ws = guarded(B, nbytes)
    x = synth.draw_x(rng, M, synth.map_size(im), dtype)
    y, ref = run_ex(B, qw, dw, x, dtype, im, 0, None, 256, workspace=ws)
    check_output(y, ref, dtype, 5e-4, "re-laid M=%d" % M)
    assert band_intact(buf, nbytes)


@pytest.mark.parametrize("M", [40, 300, 600])
def test_bf16_copy_and_split_tiles_stay_inside(B, M):
    rng = np.random.default_rng(1300 + M)
    qw = synth.draw_qweight(rng, 300, 1024)
    dw = dev_weight(qw)
    nbytes = B.workspace_bytes(M, 1024, 300)
    buf, ws = guarded(B, nbytes)
    x = synth.draw_x(rng, M, 1024, "bf16")
    for opts in ({}, {"prefill_streamk": 1, "prefill_grid": 7}, {"prefill_streamk": 1, "prefill_grid": 7, "prefill_dual": 1}):
        B.reset_options()
        for k, v in opts.items():
            B.set_option(k, v)
        y, ref = run_ex(B, qw, dw, x, "bf16", None, 1024, None, 300, workspace=ws)
        check_output(y, ref, "bf16", 5e-4, "bf16 M=%d %s" % (M, opts))
        assert band_intact(buf, nbytes), "wrote behind the workspace: bf16 M=%d %s" % (M, opts)
        assert B.workspace_status(ws) == 0


@pytest.mark.parametrize("M", [1, 5, 8, 11, 16, 64])
def test_mlp_block_stays_inside(B, M):
    _, qs, ds = draw_mlp(77, 512, 1024)
    x = synth.draw_x(np.random.default_rng(1400 + M), M, 512, "f16")
    nbytes = B.mlp_workspace_bytes(M, 512, 1024)
    buf, ws = guarded(B, nbytes)
    for k_int in (1024, 872):
        h, h_ref, y, y_ref = run_mlp(B, qs, ds, x, k_int, -1, workspace=ws)
        # (above 16 rows the block runs on the tensor cores, whose weights are rounded to fp16 first: 5e-4 there)
        check_output(h, h_ref, "f16", TOL_H if M <= 16 else 6e-4, "h M=%d" % M)
        check_output(y, y_ref, "f16", TOL_Y, "y M=%d" % M)
        assert band_intact(buf, nbytes), "wrote behind the workspace: MLP M=%d" % M


@pytest.mark.parametrize("M,dtype", [(9, "bf16"), (16, "bf16"), (12, "f16"), (16, "f16")])
def test_advertised_workspace_gives_the_bits_of_the_librarys_own(B, M, dtype):
    """Nine to sixteen rows: the kernel and the split of a tile depend on the room in the workspace; the advertised size has
    room for what the library's own buffer gives."""
    rng = np.random.default_rng(1500 + M)
    for (N, K) in ((256, 1024), (4096, 4096)):
        qw = synth.random_qweight_fast(rng, N, K)
        dw = dev_weight(qw)
        nbytes = B.workspace_bytes(M, K, N)
        buf, ws = guarded(B, nbytes)
        x = dev_x(synth.draw_x(rng, M, K, dtype), dtype)
        y = [torch.zeros((M, N), dtype=x.dtype, device="cuda") for _ in range(2)]
        for out, w in zip(y, (None, ws)):
            B.qlinear_ex(x, K, *dw[1:], None, M, K, N, None, K, None, N, out, N, workspace=w)
        assert band_intact(buf, nbytes) and B.workspace_status(ws) == 0
        assert torch.equal(y[0], y[1]), "M=%d %s %s" % (M, dtype, (N, K))


@pytest.mark.parametrize("dtype", ["f16", "bf16"])
@pytest.mark.parametrize("M", [3, 8, 16, 17, 40, 128])
@pytest.mark.parametrize("hidden,inter,k_int", [(2048, 1152, 1152), (2048, 1152, 872), (512, 2176, 1160), (512, 3200, 8), (896, 4864, 4864), (512, 1024, 870)])
def test_mlp_block_of_odd_widths_in_the_advertised_workspace(B, M, dtype, hidden, inter, k_int):
    """Widths of an odd number of groups (the down projection on a copy of its scales at the end of the workspace) and the fp16
    copy of h beside it: nothing is written behind the advertised workspace, and it has room for what the library's own buffer
    gives, bit for bit.  What the block refuses, it refuses in both."""
    rng = np.random.default_rng(M + inter + k_int)
    qg, qu, qd = (synth.random_qweight_fast(rng, n, k) for n, k in ((inter, hidden), (inter, hidden), (hidden, inter)))
    dg, du, dd = (dev_weight(q) for q in (qg, qu, qd))
    x = synth.draw_x(rng, M, hidden, dtype)
    xd = dev_x(x, dtype)
    nbytes = B.mlp_workspace_bytes(M, hidden, inter)
    buf, ws = guarded(B, nbytes)
    ldh = k_int + (-k_int) % 8
    outs = []
    for w in (None, ws):
        h, y = (torch.zeros((M, n), dtype=xd.dtype, device="cuda") for n in (ldh, hidden))
        try:
            B.mlp_swiglu(xd, hidden, *dg[1:], *du[1:], *dd[1:], M, hidden, inter, k_int, h, ldh, y, hidden, workspace=w)
            outs.append((h, y))
        except RuntimeError as e:
            assert "unsupported" in str(e)
            outs.append(None)
    assert band_intact(buf, nbytes) and B.workspace_status(ws) == 0
    if outs[0] is None:                                    # (fp16 at decode sizes: widths that are multiples of 256, k_int of 8)
        assert outs[1] is None and dtype == "f16" and M <= 16 and (hidden % 256 or inter % 256 or k_int % 8)
        return
    assert torch.equal(outs[0][0], outs[1][0]) and torch.equal(outs[0][1], outs[1][1])
    rows = sorted(set(rng.integers(0, hidden, 32).tolist() + [0, hidden - 1]))
    h_ref, y_ref = oracle.mlp_swiglu(x, dg[0], qg.scales, qg.zeros, du[0], qu.scales, qu.zeros, dd[0], qd.scales, qd.zeros, k_int,
                                     out_rows=rows, h_dtype=dtype)
    check_output(outs[0][0][:, :k_int], h_ref, dtype, 6e-4, "h")
    check_output(outs[0][1][:, torch.as_tensor(rows, device="cuda")], y_ref, dtype, TOL_Y if dtype == "f16" else 2e-3, "y")


@pytest.mark.parametrize("M", [17, 33, 128])
@pytest.mark.parametrize("k_int", [8, 200, 870])
def test_copy_of_h_from_the_gated_launch_or_from_a_pass_of_its_own(B, M, k_int):
    """bf16: one byte less than the room for the copy that the gated launch makes, and a small kernel in between makes it; same
    bits, and nothing is written behind either workspace."""
    hidden, inter = 512, 1024
    _, _, ds = draw_mlp(78, hidden, inter)
    xd = dev_x(synth.draw_x(np.random.default_rng(1600 + M), M, hidden, "bf16"), "bf16")
    relay = (M * (hidden + 8) * 2 + 255) // 256 * 256 + 512                      # what the size query of a linear adds for re-laying
    tight = (M * ((k_int + 63) // 64 * 64) * 2 + 255) // 256 * 256 + (B.workspace_bytes(M, hidden, 1) - relay) + 256
    outs = []
    for nbytes in (B.mlp_workspace_bytes(M, hidden, inter), tight, tight - 1):
        buf, ws = guarded(B, nbytes)
        h, y = (torch.zeros((M, n), dtype=xd.dtype, device="cuda") for n in (872, hidden))
        B.mlp_swiglu(xd, hidden, *ds[0][1:], *ds[1][1:], *ds[2][1:], M, hidden, inter, k_int, h, 872, y, hidden, workspace=ws)
        assert band_intact(buf, nbytes) and B.workspace_status(ws) == 0
        outs.append((h, y))
    for h, y in outs[1:]:
        assert torch.equal(h, outs[0][0]) and torch.equal(y, outs[0][1])
