"""The tcgen05 prefill attention of affine, symmetric and KIVI caches at the edges of
its 64-token tiles, their halves, and its CTAs of 256 query rows, two of which
share a tile at head_dim 128: queries in the first CTA only, one in the second,
one past a pair; tiles that end in a KIVI residual window or beyond the cache;
GQA groups that do not divide the rows; 2- and 4-bit codes.  Tolerance: the
parity bound of the other bf16 attention tests."""
import pytest
import torch

from oracle import kvq_oracle as O
from paper_2609_04263_gb300 import kvq, synth
from tests.gpu_common import require_gpu
from tests.helpers import FORMATS, check_attention, gpu_cache, kv_pair, oracle_cache

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    require_gpu()


CASES = [   # format, D, B, H, Hq, tokens, queries
    ("kivi2", 128, 1, 1, 1, 65, 65),          # one tile and a token, the first CTA only
    ("kivi2", 128, 2, 1, 4, 257, 65),         # one query in the second CTA
    ("kivi4", 128, 1, 2, 8, 400, 129),        # one past a pair
    ("kivi2", 128, 1, 1, 16, 700, 33),
    ("affine4", 128, 1, 1, 3, 300, 300),      # rows that no head fills
    ("affine2", 128, 1, 1, 2, 96, 96),        # a last tile of one half
    ("sym4", 128, 1, 2, 2, 513, 513),         # one row in the second pair
    ("sym2", 128, 1, 1, 16, 130, 17),
    ("affine4", 64, 2, 1, 8, 300, 33),
    ("kivi2", 64, 1, 2, 4, 257, 257),
    ("sym2", 64, 1, 1, 1, 31, 31),
    ("kivi4", 64, 1, 1, 5, 200, 70),
]


@pytest.mark.parametrize("fmt,D,B,H,Hq,T,L", CASES)
def test_prefill_tiles(fmt, D, B, H, Hq, T, L):
    spec = FORMATS[fmt]
    gc = gpu_cache(spec, B, H, Hq, D, T, "bf16")
    oc = oracle_cache(spec, B, H, D, T, "bf16")
    kt, vt, kn, vn = kv_pair(B, H, T, D, "bf16", seed=T + L)
    gc.append(kt, vt)
    oc.append(kn, vn)
    q = torch.from_numpy(synth.queries((B, Hq, L, D), seed=T)).to(torch.bfloat16)
    got = gc.attend_prefill(q.cuda()).float().cpu().numpy()
    assert kvq.kvq_device_status(torch.cuda.current_stream().cuda_stream) == 0
    check_attention(got, O.attend(oc, q.float().numpy()), "bf16", fmt)


@pytest.mark.parametrize("fmt,D,H,Hq", [("affine4", 128, 1, 2), ("kivi4", 128, 1, 4), ("sym4", 64, 1, 2),
                                        ("kvarn", 256, 1, 2)])
@pytest.mark.parametrize("grow", [(2, 5, 6, 9), (1, 2, 3, 4, 5, 6, 7, 8, 9), (3, 8)])
def test_prefill_growing_maxima(fmt, D, H, Hq, grow):
    """Keys whose scores grow at some tiles, at runs and gaps of odd and even length: the
    rows' maxima jump there, O is rescaled, and the waits for the P V before it fall on
    any of its barriers' phases."""
    T, spec = 640, FORMATS[fmt]
    gc = gpu_cache(spec, 1, H, Hq, D, T, "bf16")
    oc = oracle_cache(spec, 1, H, D, T, "bf16")
    kt, vt, _, _ = kv_pair(1, H, T, D, "bf16", seed=len(grow))
    f = torch.ones(T // 64)
    for i in grow:
        f[i:] *= 2.0
    kt = (kt * f.repeat_interleave(64).to(kt)[None, None, :, None]).contiguous()
    gc.append(kt, vt)
    oc.append(kt.float().cpu().numpy(), vt.float().cpu().numpy())
    q = torch.from_numpy(synth.queries((1, Hq, T, D), seed=T)).to(torch.bfloat16) * (2.0 if len(grow) < 9 else 0.05)
    got = gc.attend_prefill(q.cuda()).float().cpu().numpy()
    assert kvq.kvq_device_status(torch.cuda.current_stream().cuda_stream) == 0
    check_attention(got, O.attend(oc, q.float().numpy()), "bf16", fmt)
