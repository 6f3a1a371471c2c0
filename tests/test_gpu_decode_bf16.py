"""bf16 activations on the decode kernel (M <= 16): staged, shared, streamed and re-laid activations, the rotary
epilogue, and magnitudes that fp16 does not have."""
import numpy as np
import pytest
import torch

import oracle
from helpers import check_output, dev_weight, dev_x
from paper_2512_03383_b200 import synth

pytestmark = pytest.mark.gpu

TOL = 4e-4       # as the fp16 decode tests: the 16-bit fixed point of the activations, plus bf16's own rounding


@pytest.fixture(scope="module")
def B():
    from paper_2512_03383_b200 import binding
    yield binding
    binding.set_path(binding.PATH_AUTO)


def linear(B, qw, dw, x32, in_map, k_in):
    packed, wp, ws, wz = dw
    M, n_in = x32.shape
    xd = dev_x(x32, "bf16")
    y = torch.full((M, qw.N + 3), -77.0, device="cuda", dtype=torch.bfloat16)
    B.qlinear_ex(xd, n_in, wp, ws, wz, None, M, qw.K, qw.N, in_map, k_in, None, qw.N, y, y.stride(0))
    torch.cuda.synchronize()
    assert B.workspace_status() == 0 and (y[:, qw.N:] == -77.0).all()
    I = oracle.expand_map(in_map) if in_map else oracle.leading(k_in)
    return y[:, :qw.N], oracle.qlinear(x32, packed, qw.scales, qw.zeros, oracle.leading(qw.N), I)


@pytest.mark.parametrize("M", [1, 4, 5, 8, 9, 16])
def test_linear(B, M):
    B.set_path(B.PATH_DECODE)                       # must not be refused, re-laid maps included
    rng = np.random.default_rng(900 + M)
    qw = synth.draw_qweight(rng, 200, 2048)
    dw = dev_weight(qw)
    for in_map, k_in in ((None, 2048), (None, 1736), (None, 870), (synth.map_per_head(16, 128, 96), 0),
                         (synth.map_per_head(16, 128, 108), 0)):
        x = synth.draw_x(rng, M, synth.map_size(in_map) if in_map else k_in, "bf16")
        y, ref = linear(B, qw, dw, x, in_map, k_in)
        check_output(y, ref, "bf16", TOL, "M=%d %s %d" % (M, in_map, k_in))


@pytest.mark.parametrize("M", [2, 7, 13])
def test_qkv_rope_with_bias(B, M):
    B.set_path(B.PATH_DECODE)
    rng = np.random.default_rng(930 + M)
    hq, hkv, D, keep, K = 4, 2, 128, 84, 512
    qs = [synth.draw_qweight(rng, n * D, K) for n in (hq, hkv, hkv)]
    ds = [dev_weight(q) for q in qs]
    bias = [synth.bf16_round(rng.standard_normal(q.N).astype(np.float32)) for q in qs]
    x, pos, idx = synth.draw_x(rng, M, K, "bf16"), synth.draw_pos(rng, M), synth.draw_idx(rng, hkv, D, keep)
    out = [torch.zeros((M, n * keep), dtype=torch.bfloat16, device="cuda") for n in (hq, hkv, hkv)]
    B.qkv_rope_proj(dev_x(x, "bf16"), K, *ds[0][1:], *ds[1][1:], *ds[2][1:], *[dev_x(b, "bf16") for b in bias], M, K, hq, hkv,
                    D, keep, keep, torch.from_numpy(idx).cuda(), torch.from_numpy(pos).cuda(), 1e6, None, out[0], hq * keep,
                    out[1], hkv * keep, out[2], hkv * keep)
    torch.cuda.synchronize()
    for j, n in enumerate((hq, hkv, hkv)):
        rows = synth.map_qk_halfheads(n, D, keep) if j < 2 else synth.map_per_head(n, D, keep)
        O = oracle.expand_map(rows)
        acc = oracle.qlinear(x, ds[j][0], qs[j].scales, qs[j].zeros, O, oracle.leading(K)) + bias[j][O]
        ref = oracle.rope(acc, n, hkv, D, keep, idx, pos, 1e6) if j < 2 else acc
        check_output(out[j], ref, "bf16", TOL, "matrix %d M=%d" % (j, M))


@pytest.mark.parametrize("scale", [2.0 ** -100, 1e-30, 1e30, 2.0 ** 110])
def test_magnitudes_outside_fp16(B, scale):
    """The fixed point takes its factor from the group's own maximum: nothing saturates or is flushed."""
    B.set_path(B.PATH_AUTO)
    rng = np.random.default_rng(950)
    qw = synth.draw_qweight(rng, 72, 512)
    dw = dev_weight(qw)
    x = synth.bf16_round(synth.draw_x(rng, 3, 512, "bf16") * np.float32(scale))
    y, ref = linear(B, qw, dw, x, None, 512)
    check_output(y, ref, "bf16", TOL, "scale %g" % scale)
