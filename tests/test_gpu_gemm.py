"""The tensor-core weight-streaming GEMM against a plain fp64 matrix product of the same bf16 inputs."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

SHAPES = [  # (R, N, K): one tile / ragged N / several row paddings / deep split-K / full projection sizes / prompt chunks
    (1, 128, 64), (3, 200, 128), (5, 300, 256), (16, 1024, 512), (17, 520, 320), (40, 257, 192), (100, 1000, 512),
    (128, 384, 1024), (8, 4096, 14336), (6, 6144, 4096), (2, 32000, 4096),
    (129, 384, 512), (200, 1000, 1024), (256, 6144, 4096), (255, 4096, 14336),      # prompt-chunk row counts (256-row padding)
]


@pytest.mark.parametrize("R,N,K", SHAPES)
def test_gemm_matches_fp64_product(lib, R, N, K):
    g = torch.Generator().manual_seed(R * 1000003 + N * 101 + K)
    A = (torch.randn(R, K, generator=g) * 1.0).to(torch.bfloat16)
    W = (torch.randn(N, K, generator=g) * 0.05).to(torch.bfloat16)
    out = lib.hsd_gemm_bf16(A.cuda(), W.cuda()).cpu().numpy()
    ref = A.to(torch.float64).numpy() @ W.to(torch.float64).numpy().T
    scale = np.sqrt(K) * 0.05
    err = np.abs(out - ref).max()
    assert err < 2e-5 * scale * np.sqrt(K) + 1e-6, (err, scale)
    assert np.abs(ref).max() > 0.1 * scale


def test_gemm_is_bit_reproducible_and_row_count_independent(lib):
    # split tiles are summed in a fixed order; a row's result does not depend on how many rows ride along
    g = torch.Generator().manual_seed(5)
    A = torch.randn(8, 4096, generator=g).to(torch.bfloat16).cuda()
    W = (torch.randn(4096, 4096, generator=g) * 0.02).to(torch.bfloat16).cuda()
    a = lib.hsd_gemm_bf16(A, W)
    b = lib.hsd_gemm_bf16(A, W)
    assert torch.equal(a, b)
    one = lib.hsd_gemm_bf16(A[:1].contiguous(), W)
    assert torch.equal(one[0], a[0])


def test_gemm_rejects_bad_shapes(lib):
    A = torch.zeros(4, 100, dtype=torch.bfloat16, device="cuda")
    W = torch.zeros(64, 100, dtype=torch.bfloat16, device="cuda")
    with pytest.raises(lib.HsdError):
        lib.hsd_gemm_bf16(A, W)          # K not a multiple of 64


@pytest.mark.parametrize("R,N,K", [(24, 14257, 256),     # whole tiles of 104 rows, the last one of 9
                                   (256, 2048, 5632),    # k-blocks over a cluster of four, one accumulator buffer
                                   (5, 100, 64),         # one k-block: no split, no second accumulator
                                   (17, 1000, 192),      # three k-blocks over a cluster of two: one and two
                                   (33, 19100, 128),     # more tiles than SMs: a CTA's second tile
                                   (200, 19100, 192), (256, 57000, 128), (129, 38000, 64)])   # ... with room for one tile's accumulators
def test_gemm_tile_and_cluster_edges(lib, R, N, K):
    g = torch.Generator().manual_seed(R + N + K)
    A = torch.randn(R, K, generator=g).to(torch.bfloat16).cuda()
    W = (torch.randn(N, K, generator=g) * 0.05).to(torch.bfloat16).cuda()
    out = lib.hsd_gemm_bf16(A, W).double()
    ref = A.double() @ W.double().T
    # fp32 accumulation: 2^-23 per addition of a chain of K / 32 partial sums of this size, at most
    bound = 2.0 ** -23 * (K / 32) * (A.double().abs() @ W.double().abs().T) + 1e-7
    assert bool(((out - ref).abs() < bound).all())


@pytest.mark.parametrize("R", [33, 129])
@pytest.mark.parametrize("N,K", [(7, 64),              # a tile of 8 rows
                                 (250, 576), (1025, 1024), (1792, 512),     # clusters of eight: tiles of 24, 80 and 128 rows
                                 (1793, 512), (2048, 1088), (4097, 256),    # of four
                                 (4737, 192), (5632, 320), (9472, 128)])    # of two
def test_gemm_of_more_rows_takes_narrower_tiles_of_the_same_sums(lib, R, N, K):
    g = torch.Generator().manual_seed(R + N + K)
    A = torch.randn(R, K, generator=g).to(torch.bfloat16).cuda()
    W = (torch.randn(N, K, generator=g) * 0.05).to(torch.bfloat16).cuda()
    out = lib.hsd_gemm_bf16(A, W)
    few = torch.cat([lib.hsd_gemm_bf16(A[r:r + 32].contiguous(), W) for r in range(0, R, 32)])     # full tiles
    assert torch.equal(out, few)                          # the k-blocks are divided alike, whatever the rows of a tile
    bound = 2.0 ** -23 * (K / 32) * (A.double().abs() @ W.double().abs().T) + 1e-7
    assert bool(((out.double() - A.double() @ W.double().T).abs() < bound).all())


@pytest.mark.parametrize("R,N,K", [(5, 1024, 4096), (24, 14336, 512), (200, 2000, 1024)])
def test_gemm_calls_back_to_back_see_what_the_stream_wrote_before(lib, R, N, K):
    # a call starts under the end of the one before it: operands rewritten between calls, a result that is the next operand,
    # one workspace and one result buffer for all
    g = torch.Generator(device="cuda").manual_seed(R)
    A = [torch.randn(R, K, generator=g, device="cuda").to(torch.bfloat16) for _ in range(3)]
    W = [(torch.randn(N, K, generator=g, device="cuda") * 0.05).to(torch.bfloat16) for _ in range(3)]
    want = [lib.hsd_gemm_bf16(a, w) for a, w in zip(A, W)]
    a, w = torch.empty_like(A[0]), torch.empty_like(W[0])
    out = torch.empty(R, N, device="cuda")
    ws = torch.empty(lib.hsd_gemm_workspace_bytes(R, N, K) + 256, dtype=torch.uint8, device="cuda")
    got = []
    for i in range(24):
        a.copy_(A[i % 3])
        w.copy_(W[i % 3])
        lib.hsd_gemm_bf16(a, w, out=out, workspace=ws, check=False)
        lib.hsd_gemm_bf16(A[0], W[0], workspace=ws, check=False)
        got.append(out.clone())
    assert all(torch.equal(o, want[i % 3]) for i, o in enumerate(got))
    square = (torch.randn(K, K, generator=g, device="cuda") * 0.02).to(torch.bfloat16)
    x, y = A[0], A[0]
    for _ in range(6):
        x = lib.hsd_gemm_bf16(x, square, check=False).to(torch.bfloat16)
        y = lib.hsd_gemm_bf16(y, square).to(torch.bfloat16)
    assert torch.equal(x, y)
