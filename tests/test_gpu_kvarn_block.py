"""The KVarN block coder with the block in registers, bit for bit against the
oracle: every (head_dim, block) it is built for, 2-, 4- and 8-bit codes, and
values outside the range in which it divides by reciprocals (zero rows,
subnormal and very large activations, which take IEEE divisions)."""
import numpy as np
import pytest
import torch

from oracle import kvq_oracle as O
from tests.gpu_common import require_gpu
from tests.helpers import ACT, compare_planes, gpu_cache, kv_pair, oracle_cache

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    require_gpu()


def _spec(kb, vb, G, S):
    return dict(fmt=O.FMT_KVARN, key_bits=kb, value_bits=vb, group_size=G, sink_tokens=S,
                norm_iters=8)


@pytest.mark.parametrize("D", [64, 128, 256])
@pytest.mark.parametrize("G", [32, 64])
@pytest.mark.parametrize("kb,vb,act", [(4, 2, "bf16"), (8, 4, "bf16"), (2, 8, "f32")])
def test_every_shape(D, G, kb, vb, act):
    spec, S = _spec(kb, vb, G, 8), 8
    chunks = [S + G // 2, G, 2 * G + 1]            # a block from the staging ring, then from the input
    oc = oracle_cache(spec, 1, 3, D, sum(chunks), act)
    gc = gpu_cache(spec, 1, 3, 3, D, sum(chunks), act)
    for i, n in enumerate(chunks):
        kt, vt, kn, vn = kv_pair(1, 3, n, D, act, seed=31 + D, stream=i)
        gc.append(kt, vt)
        oc.append(kn, vn)
    compare_planes(gc, oc)


@pytest.mark.parametrize("scale", [1e-38, 1e-30, 1e-12, 1e12, 1e17])
@pytest.mark.parametrize("D,G", [(256, 64), (64, 32)])
def test_values_outside_the_reciprocal_range(scale, D, G):
    spec = _spec(4, 2, G, 0)
    L = 2 * G
    rng = np.random.default_rng(7)
    x = rng.standard_normal((2, 1, 1, L, D)).astype(np.float32)
    x[:, :, :, 3] *= np.float32(scale)             # one row far from the others
    x[:, :, :, :, 5] *= np.float32(scale)          # and one channel
    x[:, :, :, 9] = 0.0
    x[1, :, :, G:] *= np.float32(scale)            # a whole block of values
    k, v = (torch.from_numpy(t).to(ACT["f32"]) for t in x)
    oc = oracle_cache(spec, 1, 1, D, L, "f32")
    gc = gpu_cache(spec, 1, 1, 1, D, L, "f32")
    gc.append(k.cuda(), v.cuda())
    with np.errstate(all="ignore"):
        oc.append(k.numpy(), v.numpy())
    compare_planes(gc, oc)
