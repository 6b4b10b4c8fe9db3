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
