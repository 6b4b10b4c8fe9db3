"""The streaming KVarN decode at its edges: GQA groups of 1 to 8 (one or two query
columns to a lane pair), tokens that end on a block and one past it (nothing
staged, one staged token), caches whose heads span several CTAs, at both block
shapes it takes; groups of odd size, whose partials end off a 16-byte boundary,
and eight heads of 256, whose ring holds one stage only.  Tolerance: the parity bound of the other bf16 attention tests."""
import pytest

from oracle import kvq_oracle as O
from tests.gpu_common import require_gpu
from tests.helpers import FORMATS, check_attention, gpu_cache, kv_pair, oracle_cache
from tests.test_gpu_attend import _q

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    require_gpu()


CASES = [   # format, B, H, Hq, D, tokens
    ("kvarn", 16, 8, 8, 256, 128 + 64 * 10),        # group 1, nothing staged
    ("kvarn", 8, 8, 24, 256, 128 + 64 * 20 + 1),    # group 3, one staged token
    ("kvarn", 8, 8, 56, 256, 128 + 64 * 20 + 63),   # group 7, a full staging ring but one
    ("kvarn", 8, 8, 64, 256, 128 + 64 * 20),        # group 8: a ring of one stage
    ("kvarn", 3, 8, 64, 256, 128 + 64 * 61 + 5),    # its heads cut between CTAs
    ("kvarn_small", 16, 8, 8, 64, 40 + 32 * 20),
    ("kvarn_small", 16, 8, 40, 64, 40 + 32 * 20 + 1),
    ("kvarn_small", 16, 8, 64, 64, 40 + 32 * 21 - 1),
]


@pytest.mark.parametrize("fmt,B,H,Hq,D,T", CASES)
def test_stream_decode(fmt, B, H, Hq, D, T):
    gc = gpu_cache(FORMATS[fmt], B, H, Hq, D, T + 8, "bf16")
    oc = oracle_cache(FORMATS[fmt], B, H, D, T + 8, "bf16")
    kt, vt, kn, vn = kv_pair(B, H, T, D, "bf16", seed=T)
    gc.append(kt, vt)
    oc.append(kn, vn)
    qt, qn = _q(B, Hq, 1, D, "bf16", 0)
    got = gc.attend_decode(qt).float().cpu().numpy()
    check_attention(got, O.attend(oc, qn), "bf16", fmt)
