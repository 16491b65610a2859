"""Kernels that start while the one before them drains (programmatic dependent launch) read nothing that it writes: weights
written by the kernel right before the product, into the buffer that the product before has just read, and activations
that are the output of the product before.  Output, workspace and inputs exist beforehand, so that no other kernel
stands between the two."""
import pytest
import torch

import paper_2608_06763_b200 as cq

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mode", [cq.CQ_MODEL_DTYPE, cq.CQ_DYN_A8])
@pytest.mark.parametrize("M", [1, 2, 8, 16, 64])
@pytest.mark.parametrize("B,G", [(1, 128), (3, 128), (4, 128), (8, 32)])   # the first two: weights straight to registers at one token
def test_weights_written_by_the_kernel_before(B, G, M, mode):
    N, K = 2048, 4096
    L, stream = cq.lib(), torch.cuda.current_stream().cuda_stream
    g = torch.Generator(device="cuda")
    g.manual_seed(B + M)
    top = 1 if B == 1 else (1 << (B - 1)) - 1
    x = torch.randn((M, K), generator=g, device="cuda").to(torch.bfloat16)
    ws = torch.zeros(cq.cq_workspace_bytes(B, G, M, N, K, mode), dtype=torch.uint8, device="cuda")
    layout = torch.zeros(cq.cq_layout_bytes(B, G, N, K), dtype=torch.uint8, device="cuda")
    pw = cq.PackedWeights(layout, B, G, N, K)
    versions = []
    for v in range(6):
        k = torch.randint(-top, top + 1, (N, K), generator=g, device="cuda").to(torch.int8)
        k = torch.where(k == 0, torch.ones_like(k), k) if B == 1 else k
        s = 2.0 ** v * (0.5 + torch.rand((N, K // G), generator=g, device="cuda"))
        a = (0.5 + 0.5 * torch.rand((N, K // G), generator=g, device="cuda")).half()
        b = (-0.3 * torch.rand((N, K // G), generator=g, device="cuda")).half()
        codes = cq.cq_pack_codes(k, B)
        alone = cq.cq_gemm(cq.cq_repack(codes, s, a, b, B, G, N, K), x, mode, ws)
        versions.append((codes, s, a, b, alone, torch.empty_like(alone)))
    torch.cuda.synchronize()
    for _ in range(20):
        for codes, s, a, b, _, y in versions:
            assert L.cq_repack(codes.data_ptr(), s.data_ptr(), a.data_ptr(), b.data_ptr(), B, G, N, K, layout.data_ptr(), stream) == 0
            cq.cq_gemm(pw, x, mode, ws, y)
        for *_, alone, y in versions:
            assert torch.equal(y.view(torch.int16), alone.view(torch.int16))


@pytest.mark.parametrize("mode", [cq.CQ_MODEL_DTYPE, cq.CQ_DYN_A8])
@pytest.mark.parametrize("M", [1, 2, 8, 16, 64, 300])
@pytest.mark.parametrize("B,G", [(3, 128), (4, 64), (8, 32)])
def test_activations_written_by_the_kernel_before(B, G, M, mode):
    K, steps = 2048, 12
    g = torch.Generator(device="cuda")
    g.manual_seed(B + M)
    top = (1 << (B - 1)) - 1

    def matrix():
        k = torch.randint(-top, top + 1, (K, K), generator=g, device="cuda").to(torch.int8)
        s = 0.02 * (0.5 + torch.rand((K, K // G), generator=g, device="cuda"))
        a, b = torch.full_like(s, 0.8).half(), torch.full_like(s, -0.1).half()
        return cq.cq_repack(cq.cq_pack_codes(k, B), s, a, b, B, G, K, K)

    chain = [matrix() for _ in range(3)]
    x = torch.randn((M, K), generator=g, device="cuda").to(torch.bfloat16)
    ws = [torch.zeros(cq.cq_workspace_bytes(B, G, M, K, K, mode), dtype=torch.uint8, device="cuda") for _ in chain]
    ys = [torch.empty_like(x) for _ in range(steps)]
    routes = torch.arange(M, device="cuda", dtype=torch.int32)
    offset = [0, M // 2, M]

    def run(wait):
        h = x
        for i in range(steps):
            cq.cq_gemm(chain[i % 3], h, mode, ws[i % 3], ys[i])
            h = ys[i]
            if wait:
                torch.cuda.synchronize()
        r = cq.cq_gemm_routed(chain[:2], h, routes, offset, mode)   # the gather reads what the last product writes
        torch.cuda.synchronize()
        return [y.clone() for y in ys] + [r]

    alone = run(True)
    assert all(bool(torch.isfinite(y).all()) for y in alone)
    for _ in range(10):
        for y in ys:
            y.zero_()
        assert all(torch.equal(p, q) for p, q in zip(alone, run(False)))
