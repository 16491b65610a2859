"""Token tiles that are not full: the model-dtype GEMM multiplies only the columns of tokens that exist, in sixteens (a CTA pair:
thirty-twos), each CTA of a pair bringing half of them.  Row counts around those steps for the 256-token tiles of one CTA and of
a pair, the 512-token tiles (whose second half may hold no token at all), whole and shared along K."""
import pytest
import torch

import paper_2608_06763_b200 as cq
from test_gpu_small_m import check, matrix
from util import check_y

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M", [17, 48, 65, 113, 129, 144, 145, 160, 161, 225, 255, 257, 273, 300, 385, 511, 513, 545, 769])
@pytest.mark.parametrize("N,K,B,G", [(1024, 1024, 4, 128), (2888, 512, 3, 64), (6144, 2048, 8, 128)])
def test_ragged_token_tiles(N, K, B, G, M):
    check(N, K, B, G, M, cq.CQ_MODEL_DTYPE)


@pytest.mark.parametrize("M", [33, 144, 200, 300, 545])
@pytest.mark.parametrize("N,K,B,G", [(1021, 1024, 4, 128), (2885, 512, 5, 64)])   # rows of y that no 16-byte piece starts
def test_ragged_token_tiles_f16_and_odd_channels(N, K, B, G, M):
    check(N, K, B, G, M, cq.CQ_MODEL_DTYPE, torch.float16)


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float16])
@pytest.mark.parametrize("B,G", [(4, 64), (8, 128)])
def test_ragged_classes_of_the_routed_call(B, G, dtype):
    # matrices of the classes of 256 and of 512 tokens, several to a launch, each with a last tile that is not full; the columns
    # skipped in one matrix's tile are rows of the next matrix
    N, K, counts = 1048, 512, [200, 145, 300, 0, 600, 17, 256, 385]
    parts = [matrix(N, K, B, G, seed=e) for e in range(len(counts))]
    offset = [sum(counts[:e]) for e in range(len(counts) + 1)]
    g = torch.Generator(device="cuda")
    g.manual_seed(B)
    T = 700
    x = torch.randn((T, K), generator=g, device="cuda").to(dtype)
    routes = torch.randint(0, T, (offset[-1],), generator=g, device="cuda").to(torch.int32)
    y = cq.cq_gemm_routed([p[2] for p in parts], x, routes, offset).double()
    for e, (_, _, pw) in enumerate(parts):
        rows = slice(offset[e], offset[e + 1])
        if counts[e]:
            want = x[routes[rows].long()].double() @ cq.cq_decode_weights(pw).double().T
            check_y(y[rows].cpu().numpy(), want.cpu().numpy(), f"matrix {e}, {counts[e]} rows, W{B} {dtype}")
