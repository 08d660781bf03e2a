"""omq_gemm_bf16 at sizes that take each of its output tiles (single CTAs of 64, 128 and 256 columns, pairs
of 128, 192 and 256), with ragged last tiles.  Operands are small integers, so every product and sum is
exact in fp32 and the comparison is for equality.  The tile of each size is asserted, so that another cost model
cannot leave one of them untested."""
import pytest
import torch

from paper_2308_13137_gb300 import _lib

pytestmark = pytest.mark.gpu

TILES = {   # M, N, K: columns of the tile and its CTAs
    (129, 136, 72): (64, 1),
    (412, 2048, 520): (64, 1),
    (100, 8, 8): (64, 1),
    (300, 12288, 264): (128, 1),
    (120, 22016, 136): (128, 1),
    (120, 22016, 1032): (256, 1),
    (300, 4096, 200): (128, 2),
    (512, 12288, 136): (192, 2),
    (1000, 6408, 328): (192, 2),
    (1531, 4096, 776): (192, 2),
    (2048, 4104, 1024): (256, 2),
    (2048, 12288, 512): (256, 2),
    (1531, 12288, 320): (256, 2),
}


@pytest.mark.parametrize("layout", [(1, 1), (1, 0), (0, 0)])
@pytest.mark.parametrize("M,N,K", TILES)
def test_gemm_tiles(cuda_lib, M, N, K, layout):
    ak, bk = layout
    assert _lib.omq_gemm_tile(M, N, K) == TILES[M, N, K]
    if not ak and M % 8:
        M += 8 - M % 8
    g = torch.Generator(device="cuda").manual_seed(M + N + K)
    ints = lambda *s: torch.randint(-4, 5, s, generator=g, device="cuda").float()
    A, B = ints(M, K), ints(N, K)
    bias, R = ints(N), ints(M, N)
    a = (A if ak else A.T).to(torch.bfloat16).contiguous()
    b = (B if bk else B.T).to(torch.bfloat16).contiguous()
    C = torch.full((M, N), 7.0, device="cuda")
    Cb = torch.empty(M, N, device="cuda", dtype=torch.bfloat16)
    st = torch.zeros(1, dtype=torch.int32, device="cuda")
    _lib.omq_gemm_bf16(M, N, K, 1, a, K if ak else M, 0, ak, b, K if bk else N, 0, bk, C, Cb, N, 0, 1.0, bias, R, N, 0.0,
                       0, st)
    ref = (A.double() @ B.double().T + bias.double() + R.double()).float()
    torch.cuda.synchronize()
    assert int(st.item()) == 0
    assert torch.equal(C, ref) and torch.equal(Cb, ref.to(torch.bfloat16))
