"""Token tiles that are not full: the model-dtype GEMM multiplies only the columns of tokens that exist, in sixteens (a CTA pair:
thirty-twos), each CTA of a pair bringing half of them.  Row counts around those steps for the 256-token tiles of one CTA and of
a pair, the 512-token tiles (whose second half may hold no token at all), whole and shared along K."""
import pytest

import paper_2608_06763_b200 as cq
from test_gpu_small_m import check

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M", [17, 48, 65, 113, 129, 144, 145, 160, 161, 225, 255, 257, 273, 300, 385, 511, 513, 545, 769])
@pytest.mark.parametrize("N,K,B,G", [(1024, 1024, 4, 128), (2888, 512, 3, 64), (6144, 2048, 8, 128)])
def test_ragged_token_tiles(N, K, B, G, M):
    check(N, K, B, G, M, cq.CQ_MODEL_DTYPE)
