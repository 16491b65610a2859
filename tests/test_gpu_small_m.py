"""The small-M kernels where their work is cut: runs of units and tiles that end inside a strip or a row block, strips shared by
many CTAs, activations staged in parts, ragged edges, and the sizes next to the lines of the dispatch.  The reference is the
decoded matrix (cq_decode_weights, cq_decode_carriers: held to the oracle elsewhere) times the activations in fp64; the tolerance is
that of every product (util.check_y)."""
import pytest
import torch

import paper_2608_06763_b200 as cq
from util import check_y

pytestmark = pytest.mark.gpu


def matrix(N, K, B, G, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    top = 1 if B == 1 else (1 << (B - 1)) - 1
    k = torch.randint(-top, top + 1, (N, K), generator=g, device="cuda").to(torch.int8)
    if B == 1:
        k = torch.where(k == 0, torch.ones_like(k), k)
    s = 0.03 + 0.06 * torch.rand((N, K // G), generator=g, device="cuda")
    a = (0.5 + 0.5 * torch.rand((N, K // G), generator=g, device="cuda")).half()
    b = (-0.3 * torch.rand((N, K // G), generator=g, device="cuda")).half()
    return k, s, cq.cq_repack(cq.cq_pack_codes(k, B), s, a, b, B, G, N, K)


def activations(M, K, dtype, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    x = torch.randn((M, K), generator=g, device="cuda")
    x[:, :: 97] *= 20.0
    x[0, : K // 2] *= 2.0 ** -20   # tiles far apart in magnitude: each 128 k are scaled by themselves
    return x.to(dtype)


def reference(k, s, pw, x, mode):
    if mode == cq.CQ_MODEL_DTYPE:
        return x.double() @ cq.cq_decode_weights(pw).double().T
    x8, dx = cq.cq_quantize_a8(x)
    N, K, G = pw.N, pw.K, pw.G
    table = cq.cq_decode_carriers(pw).long()                                     # [N, K / G, magnitudes]
    mag = k.long().abs().view(N, K // G, G)
    c = (torch.gather(table, 2, mag if pw.B > 1 else torch.zeros_like(mag)) * k.long().sign().view(N, K // G, G)).double()
    w = (c * s.double().unsqueeze(2)).view(N, K)
    return (dx.double() / 127.0).unsqueeze(1) * (x8.double() @ w.T)


def check(N, K, B, G, M, mode, dtype=torch.bfloat16):
    k, s, pw = matrix(N, K, B, G, seed=N + K + B)
    x = activations(M, K, dtype, seed=M)
    ws = torch.zeros(cq.cq_workspace_bytes(B, G, M, N, K, mode), dtype=torch.uint8, device="cuda")
    y = cq.cq_gemm(pw, x, mode, ws).clone()
    again = cq.cq_gemm(pw, x, mode, ws)
    check_y(y.double().cpu().numpy(), reference(k, s, pw, x, mode).cpu().numpy(), f"{N}x{K} W{B} G{G} M={M} mode={mode}")
    assert torch.equal(y.view(torch.int16), again.view(torch.int16))   # partial sums added in K order, counters left at zero
    assert cq.cq_gemm_status(ws) == 0


@pytest.mark.parametrize("M", [1, 2])
@pytest.mark.parametrize("N,K,B,G", [
    (16, 32, 4, 32),          # one unit, a quarter of it real
    (1, 128, 8, 128),
    (2000, 512, 3, 64),       # whole strips, a ragged last one
    (2377, 1056, 6, 32),      # K ends inside a tile
    (300, 28672, 3, 128),     # nineteen strips shared by all SMs, eight to a strip
    (3200, 12288, 4, 128),    # runs longer than a strip that begin and end anywhere
    (3200, 12288, 1, 128),    # the same without the ring
    (512, 16384, 8, 32),      # two tokens: more than shared memory holds, the other kernel's
])
def test_strips(N, K, B, G, M):
    check(N, K, B, G, M, cq.CQ_MODEL_DTYPE, torch.float16 if N == 2000 else torch.bfloat16)


@pytest.mark.parametrize("mode", [cq.CQ_MODEL_DTYPE, cq.CQ_DYN_A8])
@pytest.mark.parametrize("M", [3, 8, 9, 16])
@pytest.mark.parametrize("N,K,B,G", [
    (100, 128, 4, 128),       # one tile
    (2816, 2048, 4, 64),      # runs that cross into the next row block
    (57344, 128, 5, 64),      # a row block is a single tile
    (8192, 8192, 8, 128),     # long runs; sixteen rows of a run do not fit shared memory at a time
    (24576, 1056, 6, 32),     # K ends inside a tile, several row blocks to a run
])
def test_row_blocks(N, K, B, G, M, mode):
    check(N, K, B, G, M, mode, torch.float16 if N == 2816 else torch.bfloat16)


def every_part_counts(N, K, B, G, M, mode, dtype, lift):
    """As check, but with sums to which every group contributes alike: plain activations, or (lift) the first half of K scaled
    down by a power of two that its group scales take back.  One power of two for a whole row of activations would leave nothing
    of that half in binary16."""
    k, s, pw = matrix(N, K, B, G, seed=N + K + B)
    g = torch.Generator(device="cuda")
    g.manual_seed(M)
    x = torch.randn((M, K), generator=g, device="cuda")
    if lift:
        down, groups = 2.0 ** -34 if dtype == torch.bfloat16 else 2.0 ** -12, K // G // 2
        x[:, : groups * G] *= down
        s = s.clone()
        s[:, :groups] /= down
        codes, _, a, b = cq.cq_unpack(pw)
        pw = cq.cq_repack(codes, s, a, b, B, G, N, K)
    x = x.to(dtype)
    ws = torch.zeros(cq.cq_workspace_bytes(B, G, M, N, K, mode), dtype=torch.uint8, device="cuda")
    y = cq.cq_gemm(pw, x, mode, ws)
    check_y(y.double().cpu().numpy(), reference(k, s, pw, x, mode).cpu().numpy(), f"{N}x{K} W{B} G{G} M={M} mode={mode} lift={lift}")


@pytest.mark.parametrize("lift", [False, True])
@pytest.mark.parametrize("M", [1, 2])
@pytest.mark.parametrize("N,K,B,G", [
    (2000, 512, 3, 64), (2377, 1056, 6, 32),
    (300, 28672, 1, 128), (300, 28672, 3, 128), (300, 28672, 2, 64),            # shared strips, at one token without the ring and with it
    (3200, 12288, 1, 128), (3200, 12288, 2, 128), (3200, 12288, 3, 128), (3200, 12288, 4, 128), (3200, 12288, 8, 32),
    (5248, 1280, 7, 64),                                                         # whole strips, three on some SMs
])
def test_strips_every_part_counts(N, K, B, G, M, lift):
    every_part_counts(N, K, B, G, M, cq.CQ_MODEL_DTYPE, torch.float16 if N == 2000 else torch.bfloat16, lift)


@pytest.mark.parametrize("mode,lift", [(cq.CQ_MODEL_DTYPE, False), (cq.CQ_MODEL_DTYPE, True), (cq.CQ_DYN_A8, False)])
@pytest.mark.parametrize("M", [3, 8, 16])
@pytest.mark.parametrize("N,K,B,G", [
    (100, 384, 4, 128),                                                          # a tile each to CTAs of one set
    (2048, 1024, 5, 128), (2304, 1024, 4, 64), (4736, 1024, 3, 128),             # just below one and two tiles an SM, and at two
    (2816, 2048, 4, 64), (8192, 8192, 8, 128), (24576, 1056, 6, 32),
])
def test_row_blocks_every_part_counts(N, K, B, G, M, mode, lift):
    every_part_counts(N, K, B, G, M, mode, torch.float16 if N == 2816 else torch.bfloat16, lift)
