"""The tcgen05 prefill attention of KVarN caches (head_dim 256, 64-token blocks)
at the edges of its 64-token tiles, their 32-token halves and the pairs of
128-row CTAs: sinks only, sinks that end inside a tile, the first coded block,
staged tokens, a chunk of queries at the end of a longer cache, queries in the
first CTA only and one in the second, GQA groups that do not divide the rows,
2- and 4-bit codes.  Tolerance: the
parity bound of the other bf16 attention tests."""
import numpy as np
import pytest
import torch

from oracle import kvq_oracle as O
from paper_2609_04263_gb300 import kvq, synth
from tests.gpu_common import require_gpu
from tests.helpers import gpu_cache, kv_pair, oracle_cache

pytestmark = pytest.mark.gpu
D = 256


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    require_gpu()


CASES = [   # kb, vb, sinks, B, H, Hq, tokens, queries
    (4, 2, 128, 1, 1, 1, 1, 1),
    (4, 2, 128, 1, 1, 2, 18, 18),       # the last call of the other kernel, the first of this one
    (4, 2, 128, 1, 1, 2, 19, 18),
    (4, 4, 0, 2, 1, 1, 66, 1),
    (4, 2, 128, 1, 1, 2, 32, 32),
    (4, 2, 128, 2, 1, 2, 129, 129),
    (4, 2, 128, 1, 2, 4, 192, 192),
    (4, 2, 128, 1, 2, 4, 255, 65),
    (4, 2, 128, 1, 1, 3, 400, 400),
    (4, 2, 128, 1, 1, 16, 321, 9),
    (4, 2, 128, 2, 2, 4, 1500, 300),
    (4, 4, 0, 1, 1, 2, 200, 200),
    (2, 2, 32, 1, 2, 4, 500, 77),
    (2, 4, 64, 1, 1, 2, 130, 130),
    (4, 2, 96, 2, 1, 1, 300, 129),
    (2, 2, 64, 1, 1, 1, 257, 257),
    (4, 4, 32, 1, 2, 2, 1025, 128),
    (4, 2, 40, 1, 1, 2, 200, 200),      # sinks off the tile: the other kernel
]


@pytest.mark.parametrize("kb,vb,S,B,H,Hq,T,L", CASES)
def test_prefill_parity(kb, vb, S, B, H, Hq, T, L):
    spec = dict(fmt=O.FMT_KVARN, key_bits=kb, value_bits=vb, group_size=64, sink_tokens=S, norm_iters=8)
    gc = gpu_cache(spec, B, H, Hq, D, T, "bf16")
    oc = oracle_cache(spec, B, H, D, T, "bf16")
    kt, vt, kn, vn = kv_pair(B, H, T, D, "bf16", seed=T + L)
    gc.append(kt, vt)
    oc.append(kn, vn)
    q = torch.from_numpy(synth.queries((B, Hq, L, D), seed=T)).to(torch.bfloat16)
    got = gc.attend_prefill(q.cuda()).float().cpu().numpy()
    assert kvq.kvq_device_status(torch.cuda.current_stream().cuda_stream) == 0
    err = np.abs(got - O.attend(oc, q.float().numpy())).max()
    assert err <= 2e-2, f"max-abs {err}"


def _one_query(gc, Q):
    """The newest token's query Q e_1 (rotated: Q / 16 with alternating signs), at scale 1:
    the output's channel 0 over 16."""
    q = torch.zeros(1, 1, 1, D)
    q[..., 1] = Q
    return gc.attend_prefill(q.bfloat16().cuda(), scale=1.0).float().cpu().numpy()[0, 0, 0, 0] / 16


def test_full_precision_key_bits():
    """A sink's key keeps 16 bits and more beside a bf16 high part that is rounded: its
    rotated channels are (1 +- b +- g) / 16 with b = 255 2^-15 and g = 2^-16, and a
    query that sees g alone has the score 2^16 g = 1 against 0 of 39 zero keys.
    After a truncated high part the remainder b +- g needs nine bits, and the
    score comes out as 1.5.  The bound is bf16's of the output."""
    gc = gpu_cache(dict(fmt=O.FMT_KVARN, key_bits=4, value_bits=2, group_size=64, sink_tokens=128,
                        norm_iters=8), 1, 1, 1, D, 40, "bf16")
    k, v = torch.zeros(1, 1, 40, D), torch.zeros(1, 1, 40, D)
    k[0, 0, 7, 0], k[0, 0, 7, 2], k[0, 0, 7, 1] = 1.0, 255 * 2.0 ** -15, 2.0 ** -16
    v[0, 0, 7, 0] = 16.0
    gc.append(k.bfloat16().cuda(), v.bfloat16().cuda())
    want = 1 / (1 + 39 * np.exp(-1.0))
    assert abs(_one_query(gc, 2.0 ** 16) - want) <= 2 ** -8 * want


def test_coded_key_bits():
    """The same of coded keys: two tokens of one block with equal scores, 543.  One key is
    r c_j with factors whose product a truncated high part and a bf16 remainder hold
    2^-16 off (score 1 off), a rounded one exactly; the other's group
    offsets (52, 60, 64, 72 / 1024 above 1, mean 62) are exact either way.  The
    block's other keys are zero."""
    gc = gpu_cache(dict(fmt=O.FMT_KVARN, key_bits=4, value_bits=2, group_size=64, sink_tokens=0,
                        norm_iters=8), 1, 1, 1, D, 64, "bf16")
    kt, vt, _, _ = kv_pair(1, 1, 64, D, "bf16", seed=1)
    gc.append(kt, vt)
    pl = gc.planes()
    for n in ("k_codes", "k_scale", "k_row", "v_codes", "v_scale", "v_row"):
        pl[n].zero_()
    for n in ("k_zero", "v_zero", "v_col"):
        pl[n].fill_(1.0)
    pl["k_col"][..., 0::2] = 1 + 24 / 1024
    pl["k_col"][..., 1::2] = 1 + 8 / 1024
    rows = pl["k_row"].view(-1)
    rows[0] = 1 + 62 / 1024
    rows[1] = 1.0
    pl["k_zero"][0, 0, 1] = 1 + torch.tensor([52.0, 60.0, 64.0, 72.0]) / 1024
    pl["v_row"].view(-1)[0] = 1.0
    assert abs(_one_query(gc, 2.0 ** 12) - 0.5) <= 2 ** -8 * 0.5
