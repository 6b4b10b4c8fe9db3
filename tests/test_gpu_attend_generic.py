"""The fp32 attention kernel (prefill and decode) at the edges of its 64-token
tiles, 16- and 64-row CTAs and decode splits, against the oracle.  Tolerance:
the parity bound of the other attention tests, 1e-4 (fp32) and 2e-2 (bf16)."""
import numpy as np
import pytest
import torch

from oracle import kvq_oracle as O
from paper_2609_04263_gb300 import synth
from tests.gpu_common import require_gpu
from tests.helpers import ACT, FORMATS, gpu_cache, kv_pair, oracle_cache

pytestmark = pytest.mark.gpu
TOL = {"f32": 1e-4, "bf16": 2e-2}


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    require_gpu()


def _caches(name, act, B, H, Hq, D, T):
    gc = gpu_cache(FORMATS[name], B, H, Hq, D, T, act)
    oc = oracle_cache(FORMATS[name], B, H, D, T, act)
    kt, vt, kn, vn = kv_pair(B, H, T, D, act, seed=T + D)
    gc.append(kt, vt)
    oc.append(kn, vn)
    return gc, oc


def _check(gc, oc, B, Hq, L, D, act, decode):
    q = torch.from_numpy(synth.queries((B, Hq, L, D), seed=L)).to(ACT[act])
    run = gc.attend_decode if decode else gc.attend_prefill
    got = run(q.cuda()).float().cpu().numpy()
    again = run(q.cuda()).float().cpu().numpy()    # the decode merge leaves its counters ready
    assert np.array_equal(got, again)
    err = np.abs(got - O.attend(oc, q.float().numpy())).max()
    assert err <= TOL[act], f"max-abs {err}"


@pytest.mark.parametrize("name,D", [("affine4", 64), ("sym8", 128), ("float", 256), ("kivi2", 128),
                                    ("kivi_k8", 64), ("kvarn", 256), ("kvarn_small", 64)])
@pytest.mark.parametrize("B,H,Hq,T,L", [(1, 1, 1, 1, 1), (1, 2, 2, 65, 65), (2, 1, 3, 200, 17),
                                        (1, 1, 16, 130, 5)])
def test_prefill(name, D, B, H, Hq, T, L):
    gc, oc = _caches(name, "f32", B, H, Hq, D, T)
    _check(gc, oc, B, Hq, L, D, "f32", False)


def test_prefill_64_row_ctas():
    """Enough rows for two 64-row CTAs per SM (4 x 8 heads x 640 queries)."""
    gc, oc = _caches("affine4", "f32", 4, 8, 8, 64, 640)
    _check(gc, oc, 4, 8, 640, 64, "f32", False)


@pytest.mark.parametrize("name,act,D", [("affine4", "f32", 64), ("kvarn", "f32", 256),
                                        ("float", "bf16", 256), ("affine8", "bf16", 64),
                                        ("kivi_r0", "f32", 128)])
@pytest.mark.parametrize("B,H,Hq,T", [(1, 4, 4, 1), (2, 2, 4, 33), (1, 1, 16, 1000), (3, 1, 5, 2049)])
def test_decode(name, act, D, B, H, Hq, T):
    gc, oc = _caches(name, act, B, H, Hq, D, T)
    _check(gc, oc, B, Hq, 1, D, act, True)


@pytest.mark.parametrize("decode", [False, True])
def test_infinite_scale(decode):
    """A symmetric group whose scale is beyond fp16 stores an infinite scale, and its
    value is an infinity of the code's sign (the channels' codes here are all
    below zero): so is the output, and the other channels are what they were."""
    D, T = 64, 5
    gc = gpu_cache(FORMATS["sym4"], 1, 1, 1, D, T, "f32")
    kt, vt, _, _ = kv_pair(1, 1, T, D, "f32", seed=3)
    vt[..., 32:] = -1e6
    gc.append(kt, vt)
    assert torch.isinf(gc.planes()["v_scale"][0, 0, :T, 1]).all()
    q = torch.from_numpy(synth.queries((1, 1, 1, D), seed=2)).cuda()
    got = (gc.attend_decode if decode else gc.attend_prefill)(q)[0, 0, 0]
    assert torch.isneginf(got[32:]).all() and torch.isfinite(got[:32]).all()


@pytest.mark.parametrize("name", ["float", "kivi2"])
def test_infinite_later_value(name):
    """Queries whose CTA ends before a token do not read its value, also where the
    number of keys they see is no multiple of 4."""
    D, T, L, t_inf = 64, 207, 200, 135            # the 128th query is at position 134
    gc = gpu_cache(FORMATS[name], 1, 1, 1, D, T, "f32")
    kt, vt, _, _ = kv_pair(1, 1, T, D, "f32", seed=5)
    vt[:, :, t_inf:] = float("inf")
    gc.append(kt, vt)
    q = torch.from_numpy(synth.queries((1, 1, L, D), seed=6)).cuda()
    assert torch.isfinite(gc.attend_prefill(q)[:, :, :128]).all()
