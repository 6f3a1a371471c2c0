"""Argument handling of the C extension behind the hot entry points (no device work: every call fails first)."""
import pytest
import torch

from paper_2512_03383_b200 import binding as B

X = torch.zeros((4, 128), dtype=torch.float16)
W = torch.zeros((16, 64), dtype=torch.uint8)
S = torch.zeros((16, 1), dtype=torch.float16)


@pytest.mark.parametrize("call, error, text", [
    (lambda: B.qlinear(X, W, S, S, 1, 100, 16, 100, 16, X, stream=0), B.UniqlError, "bad shape"),
    (lambda: B.qlinear(x=None, packed_w=W, scales=S, zeros=S, M=1, K=128, N=16, k_in=128, k_out=16, y=X, stream=0),
     B.UniqlError, "null pointer"),
    (lambda: B.qlinear(X, W, S, S, 1, 128, 16, 128, 16), TypeError, "'y'"),
    (lambda: B.qlinear(X, W, S, S, 1, 128, 16, 128, 16, X, 0, 0), TypeError, "at most 11"),
    (lambda: B.qlinear(X, W, S, S, 1, 128, 16, 128, 16, X, x=X), TypeError, "multiple values"),
    (lambda: B.qlinear(X, W, S, S, 1, 128, 16, 128, 16, X, streem=0), TypeError, "streem"),
    (lambda: B.qlinear(X, W, S, S, "1", 128, 16, 128, 16, X, 0), TypeError, "'M'"),
    (lambda: B.qlinear(X, W, S, S, 1 << 40, 128, 16, 128, 16, X, 0), OverflowError, "'M'"),
    (lambda: B.qlinear_ex(X.float(), 128, W, S, S, None, 1, 128, 16, None, 128, None, 16, X, 16, stream=0), TypeError,
     "float16 or bfloat16"),
    (lambda: B.qlinear_ex(X, 128, W, S, S, None, 1, 128, 16, [(0, 4, 4)], 0, None, 16, X, 16, stream=0), ValueError, "family"),
    (lambda: B.qlinear_ex(X, 128, W, S, S, None, 1, 128, 16, [(0, 8, 4, 1)] * 9, 0, None, 16, X, 16, stream=0), ValueError, "8"),
    (lambda: B.qlinear_ex(X, 64, W, S, S, None, 1, 128, 16, [(0, 128, 128, 1)], 0, None, 16, X, 16, stream=0), B.UniqlError,
     "bad shape"),
    (lambda: B.qlinear_multi(X, 128, 1, 128, None, 128, [{"scales": S}], stream=0), KeyError, "packed_w"),
    (lambda: B.mlp_swiglu(X, 128, W, S, S, W, S, S, W, S, S, 1, 128, 128, 128, X.bfloat16(), 128, X, 128), TypeError, "same type"),
])
def test_wrong_arguments(call, error, text):
    with pytest.raises(error, match=text):
        call()


def test_status_travels_with_the_error():
    with pytest.raises(B.UniqlError) as e:
        B.embed_rows(W, S, S, torch.zeros(2, dtype=torch.int32), X[:, :64].contiguous(), stream=0)      # rows narrower than K
    assert e.value.status == 2


@pytest.mark.parametrize("fn, written", [
    (lambda y, w: B.qlinear(X, W, S, S, 1, 100, 16, 100, 16, y, stream=0), 1),
    (lambda y, w: B.qlinear_noalloc(X, W, S, S, 1, 100, 16, 100, 16, y, stream=0), 1),
    (lambda y, w: B.qlinear_ex(X, 128, W, S, S, None, 1, 100, 16, None, 100, None, 16, y, 16, workspace=w, stream=0), 2),
    (lambda y, w: B.qlinear_multi(X, 128, 1, 100, None, 100, [dict(packed_w=W, scales=S, zeros=S, N=16, k_out=16, y=y, ldy=16)],
                                  workspace=w, stream=0), 2),
    (lambda y, w: B.qk_rope_proj(X, 128, W, S, S, W, S, S, None, None, 1, 100, 1, 1, 16, 16, S, S, 1e4, None, y, 16, w, 16, stream=0), 2),
    (lambda y, w: B.qkv_rope_proj(X, 128, W, S, S, W, S, S, W, S, S, None, None, None, 1, 100, 1, 1, 16, 16, 16, S, S, 1e4, None, y, 16,
                                  y, 16, w, 16, stream=0), 2),
    (lambda y, w: B.mlp_swiglu(X, 128, W, S, S, W, S, S, W, S, S, 0, 128, 128, 128, y, 128, w, 128, stream=0), 2),
    (lambda y, w: B.mlp_swiglu_decode(X, 128, W, S, S, W, S, S, W, S, S, 0, 128, 128, 128, y, 128, w, 128, stream=0), 2),
    (lambda y, w: B.embed_rows(W, S, S, torch.zeros(2, dtype=torch.int32), y.view(8, 64), bad_id=w, stream=0), 2),   # rows narrower than K
])
def test_written_tensors_own_their_storage(fn, written):
    """A lazy clone shares its storage until it is written to: what a call writes must not land in the tensor it was cloned
    from.  (Every call here is refused for its shapes, after its addresses were taken.)"""
    for w_only in range(written):
        y, w = torch._lazy_clone(X), torch._lazy_clone(X)
        with pytest.raises(B.UniqlError) as e:
            fn(y, w)
        assert e.value.status == 2             # (refused by the host, with or without a GPU: the addresses are the CPU's)
        assert not torch._C._is_cow_tensor(w if w_only else y)
