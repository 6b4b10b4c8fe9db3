"""The projection's tile of two CTAs (256 rows of x by 128 or 256 features) at
its edges, against the oracle: rows that end in the first CTA, on the boundary
between the two, and one past a tile; K-slices fewer than the ring's stages, one
more, and many; ranks from 0 to 64, whose A_p rows are split between the CTAs;
dense and NF4 bases.  Tolerance per (sequence, head), as for every bf16
projection: 1e-2 of the head's largest oracle value."""
import pytest

from oracle import kvq_oracle as O
from tests.gpu_common import require_gpu
from tests.helpers import check_projection
from tests.test_gpu_project import _case
from tests.test_gpu_project_nf4 import _case as _nf4_case

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    require_gpu()


# B, L, d_in, Hq, Hkv, D, ranks (q, k, v)
CASES = [
    (1, 17, 64, 2, 2, 64, (8, 8, 8)),           # one K-slice, one CTA's rows only
    (1, 127, 256, 4, 2, 64, (16, 0, 64)),       # a row short of the first CTA
    (1, 128, 320, 4, 4, 64, (24, 40, 16)),      # the ring filled once
    (3, 43, 384, 2, 2, 128, (64, 64, 64)),      # 129 rows: one in the second CTA; a slice more than the ring
    (1, 255, 512, 4, 2, 128, (0, 0, 0)),
    (2, 128, 192, 8, 4, 128, (8, 16, 24)),      # one tile exactly
    (1, 257, 448, 3, 1, 128, (32, 8, 48)),      # one row in the second tile; an odd number of heads
    (1, 513, 256, 2, 1, 256, (16, 32, 0)),      # a head as wide as the tile
    (1, 300, 4096, 32, 8, 128, (16, 16, 16)),
]


@pytest.mark.parametrize("B,L,d_in,Hq,Hkv,D,ranks", CASES)
def test_pair_tile(B, L, d_in, Hq, Hkv, D, ranks):
    from paper_2609_04263_gb300 import api
    (tx, tw, tl), (nx, nw, nl) = _case("bf16", B, L, d_in, Hq, Hkv, D, ranks)
    got = api.project_lora(tx, tw, tl, 2.0, Hq, Hkv, D, pos0=11, rope_base=10000.0)
    ref = O.project_lora(nx, nw, nl, 2.0, Hq, Hkv, D, pos0=11, rope_base=10000.0)
    for name, g, r in zip("qkv", got, ref):
        check_projection(g.float().cpu().numpy(), r, "bf16", name)


@pytest.mark.parametrize("B,L,d_in,Hq,Hkv,D,ranks", [c for c in CASES if c[5] <= 128])   # NF4 heads
def test_pair_tile_nf4(B, L, d_in, Hq, Hkv, D, ranks):
    from paper_2609_04263_gb300 import api
    (tx, tc, ta, tl), (nx, codes, absmax, nl) = _nf4_case(B, L, d_in, Hq, Hkv, D, ranks)
    got = api.project_lora_nf4(tx, tc, ta, tl, 2.0, Hq, Hkv, D, pos0=11, rope_base=10000.0)
    ref = O.project_lora_nf4(nx, codes, absmax, nl, 2.0, Hq, Hkv, D, pos0=11, rope_base=10000.0)
    for name, g, r in zip("qkv", got, ref):
        check_projection(g.float().cpu().numpy(), r, "bf16", name)
