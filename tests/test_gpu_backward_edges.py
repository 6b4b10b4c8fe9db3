"""The straight-through backward's products at the edges of their 64 x 64 tiles of 32
k, and of its softmax's key ranges: one query; stacked rows and keys a row short
of a tile, a whole one and a row past it; tiles that end with a head and tiles that
hold two, over no earlier keys and some; key counts that no vector load divides;
head_dim 64 to 256; adapters of unlike ranks (whose products share a launch); the
workspace's size; infinite values.  The checks and tolerances are those of the
other backward tests."""
import pytest
import torch

from tests import test_gpu_backward as TB
from tests.gpu_common import require_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    require_gpu()


@pytest.mark.parametrize("fmt,act,B,Hkv,Hq,D,T0,L", [
    ("affine4", "bf16", 1, 1, 1, 64, 0, 1),
    ("affine4", "f32", 1, 1, 1, 64, 3, 127),
    ("sym2", "bf16", 1, 1, 3, 128, 2, 43),       # 129 stacked rows, 45 keys
    ("kivi2", "bf16", 1, 2, 2, 64, 126, 3),
    ("affine2", "f32", 2, 1, 2, 128, 0, 65),     # 130 stacked rows
    ("affine4", "bf16", 1, 1, 2, 256, 1, 130),
    ("affine4", "f32", 1, 1, 1, 64, 0, 63),
    ("affine4", "f32", 1, 1, 1, 64, 0, 64),      # one tile of rows, one of keys
    ("sym2", "bf16", 1, 1, 1, 128, 0, 65),
    ("affine4", "f32", 1, 2, 2, 64, 64, 64),     # 128 keys
    ("affine4", "bf16", 1, 1, 2, 64, 0, 64),     # a head ends with its tile
    ("affine4", "f32", 1, 1, 2, 64, 5, 64),      # the same past earlier keys
    ("affine4", "bf16", 1, 1, 2, 64, 0, 32),     # two heads in a tile
    ("affine4", "f32", 1, 1, 4, 64, 33, 32),
    ("kivi2", "bf16", 1, 1, 2, 128, 32, 32),     # two heads in a tile, 64 keys
])
def test_attend_backward_tiles(fmt, act, B, Hkv, Hq, D, T0, L):
    TB.test_attend_backward_parity(fmt, act, B, Hkv, Hq, D, T0, L)


@pytest.mark.parametrize("act,B,L,d_in,Hq,Hkv,D,ranks,extra,pos0,base", [
    ("bf16", 1, 1, 256, 2, 2, 64, (8, 64, 16), 0, 7, 10000.0),
    ("bf16", 1, 129, 320, 4, 1, 64, (64, 0, 8), 3, 0, 10000.0),
    ("f32", 1, 127, 192, 2, 2, 128, (0, 40, 8), 0, 1, 500000.0),
    ("bf16", 1, 257, 640, 2, 2, 128, (0, 0, 16), 0, 0, 0.0),
    ("f32", 1, 66, 192, 2, 1, 64, (5, 33, 64), 0, 0, 10000.0),    # d_x over ranks no K tile divides
])
def test_lora_backward_tiles(act, B, L, d_in, Hq, Hkv, D, ranks, extra, pos0, base):
    TB.test_lora_backward_parity(act, B, L, d_in, Hq, Hkv, D, ranks, extra, pos0, base)


@pytest.mark.parametrize("L", [44, 45, 46, 47])
def test_attend_backward_workspace(L):
    """One pair's workspace is its K, V reconstruction and its S and dP, nothing more,
    whatever the number of keys is a multiple of; gradients in exactly that are those
    in one with room for padded rows."""
    from paper_2609_04263_gb300 import kvq
    B, Hkv, Hq, D, T0 = 1, 1, 3, 64, 20
    gc, _ = TB._filled(TB.FORMATS["affine4"], "bf16", B, Hkv, Hq, D, T0, L, seed=L)
    T = T0 + L
    want = (2 * T * D + 2 * (Hq // Hkv) * L * T) * 4
    per = kvq.kvq_attend_backward_workspace(gc.handle, L, Hq)
    assert per == (want + 255) // 256 * 256
    gen = torch.Generator("cuda").manual_seed(L)
    q, do = (torch.randn(B, Hq, L, D, generator=gen, device="cuda").bfloat16() for _ in range(2))
    tight = gc.attend_backward(q, do, workspace=torch.empty(per, dtype=torch.uint8, device="cuda"))
    assert all(torch.equal(a, b) for a, b in zip(tight, gc.attend_backward(q, do)))
    TB.test_attend_backward_parity("affine4", "bf16", B, Hkv, Hq, D, T0, L)


def test_attend_backward_many_pairs():
    """More (sequence, kv head) pairs than one launch of paired products has grid
    slices for (32,767), against fp64 autograd."""
    B, H, L, D, scale = 33000, 1, 3, 64, 0.125
    gc = TB.gpu_cache(TB.FORMATS["float"], B, H, H, D, L, "f32")
    gen = torch.Generator("cuda").manual_seed(4)
    q, k, v, do = (torch.randn(B, H, L, D, generator=gen, device="cuda") for _ in range(4))
    gc.append(k, v)
    got = gc.attend_backward(q, do, scale=scale)
    ref = [t.double().requires_grad_() for t in (q, k, v)]
    s = ref[0] @ ref[1].transpose(-1, -2) * scale
    s = s.masked_fill(torch.ones(L, L, dtype=torch.bool, device="cuda").triu(1), float("-inf"))
    (s.softmax(-1) @ ref[2]).backward(do.double())
    for g, r, what in zip(got, ref, ("dq", "dk", "dv")):
        TB._close(g.cpu().numpy(), r.grad.cpu().numpy(), what)


@pytest.mark.parametrize("T", [20, 21])
def test_attend_backward_infinite_scores(T):
    """Keys whose scores lie below fp32 (-9e38) have weight 0: they are the first of
    a lane's keys, four at a time (T = 20) and one at a time."""
    D, L, scale = 64, 16, 0.125
    n = T - L
    gc = TB.gpu_cache(TB.FORMATS["float"], 1, 1, 1, D, T, "f32")
    gen = torch.Generator("cuda").manual_seed(T)
    q, k, v, do = (torch.randn(1, 1, x, D, generator=gen, device="cuda") for x in (L, T, T, L))
    k[..., 0] = 0
    k[0, 0, :n] = 0
    k[0, 0, :n, 0] = -3e19
    q[..., 0] = 3e19
    gc.append(k, v)
    got = gc.attend_backward(q, do, scale=scale)
    ref = [t.double().requires_grad_() for t in (q, k, v)]
    s = ref[0] @ ref[1].transpose(-1, -2) * scale
    s = s.masked_fill(torch.ones(L, T, dtype=torch.bool, device="cuda").triu(n + 1), float("-inf"))
    (s.softmax(-1) @ ref[2]).backward(do.double())
    # (d_k's channel 0 is a sum over the queries' 3e19)
    for g, r, what in zip((got[0], got[1][..., 1:], got[2]),
                          (ref[0].grad, ref[1].grad[..., 1:], ref[2].grad), ("dq", "dk", "dv")):
        TB._close(g.cpu().numpy(), r.cpu().numpy(), what)


def test_attend_backward_infinite_key():
    """A key with an infinite channel, of scores -inf, has weight 0: all gradients but
    d_q's along that channel (0 times the key's infinity) are what they are for a
    key of large scores.  Both of the last query's tiles of 32 keys hold others."""
    D, T, L, scale = 64, 70, 66, 0.125
    gen = torch.Generator("cuda").manual_seed(1)
    q, k, v, do = (torch.randn(1, 1, x, D, generator=gen, device="cuda") for x in (L, T, T, L))
    q[..., 5] = q[..., 5].abs() + 0.1
    out = []
    for big in (float("-inf"), -1e6):
        k[0, 0, 2, 5] = big
        gc = TB.gpu_cache(TB.FORMATS["float"], 1, 1, 1, D, T, "f32")
        gc.append(k, v)
        out.append(gc.attend_backward(q, do, scale=scale))
    for g, r, what in zip(out[0], out[1], ("dq", "dk", "dv")):
        if what == "dq":
            g[..., 5] = r[..., 5] = 0
        TB._close(g.cpu().numpy(), r.double().cpu().numpy(), what)


def test_lora_backward_unaligned_dx():
    """d_x off a 16-byte boundary, at a shape whose d_x would go to the tensor cores."""
    from paper_2609_04263_gb300 import kvq
    L, d_in, Hq, Hkv, D = 70, 256, 2, 1, 64
    gen = torch.Generator("cuda").manual_seed(3)
    x, w = (torch.randn(*n, generator=gen, device="cuda").bfloat16() for n in ((L, d_in), (256, d_in)))
    dq, dk, dv = (torch.randn(1, h, L, D, generator=gen, device="cuda") for h in (Hq, Hkv, Hkv))
    n = kvq.kvq_lora_backward_workspace(1, L, d_in, Hq, Hkv, D, 0, 0, 0)
    ws = torch.empty(n, dtype=torch.uint8, device="cuda")
    dx = torch.empty(L * d_in + 1, device="cuda")[1:]
    kvq.kvq_lora_backward(x.data_ptr(), 1, L, d_in, w.data_ptr(), *(None, None, 0) * 3, 1.0, Hq, Hkv, D, 0,
                          0.0, kvq.KVQ_BF16, dq.data_ptr(), dk.data_ptr(), dv.data_ptr(), L, *(None,) * 6,
                          dx.data_ptr(), ws.data_ptr(), n, torch.cuda.current_stream().cuda_stream)
    g = torch.cat((dq, dk, dv), 1)[0].transpose(0, 1).reshape(L, -1).double()
    TB._close(dx.view(1, 1, L, d_in).cpu().numpy(), (g @ w.double())[None, None].cpu().numpy(), "d_x")
