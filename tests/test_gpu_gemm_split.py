"""The dual GEMM's split of K over a cluster: every tile width (16 to 128) and split (2, 4),
rows and columns that end inside a tile, and outputs whose rows are not 16-byte aligned,
against float64 products of the same bf16 operands.

Tolerance: the tensor cores' float32 accumulation errs in proportion to the length of the
sum (2.1e-6 of the result at two products of K = 1000, 6.5e-6 at K = 2960), so 3e-5 at the
K = 4096 and up to three products used here.
"""
import pytest

from gpu_util import need_gpu, rel_l2

SHAPES = [(1, 16, 2048), (129, 30, 1024), (256, 1000, 1024), (100, 200, 4096),
          (640, 384, 2112), (127, 64, 520)]


@pytest.mark.gpu
@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("mask", [1, 1 | 8 | 16, 2 | 4])
@pytest.mark.parametrize("pad", [0, 3])
def test_split_k(shape, mask, pad):
    torch, native = need_gpu()
    M, N, K = shape
    g = torch.Generator(device="cuda").manual_seed(M + 3 * N + 5 * K + mask)
    mk = lambda r: torch.randn(r, K, generator=g, device="cuda").to(torch.bfloat16)
    A, B = [mk(M), mk(M)], [mk(N), mk(N)]
    C = [torch.full((M, N + pad), float("nan"), device="cuda") for _ in range(2)]
    bias = [torch.randn(N, generator=g, device="cuda") for _ in range(2)]
    native.mf_dual_gemm_bf16(M, N, K, A[0], A[1], B[0], B[1], C[0], C[1], mask, *bias)
    torch.cuda.synchronize()
    terms = {1: (0, 0, 0), 2: (0, 1, 0), 4: (0, 0, 1), 8: (1, 1, 0), 16: (1, 0, 1)}
    for j in range(2):
        used = [(a, b) for bit, (c, a, b) in terms.items() if mask & bit and c == j]
        if not used:
            assert torch.isnan(C[j]).all()
            continue
        ref = sum(A[a].double() @ B[b].double().t() for a, b in used) + bias[j].double()
        assert rel_l2(C[j][:, :N].cpu(), ref.cpu()) < 3e-5
        assert pad == 0 or torch.isnan(C[j][:, N:]).all()
