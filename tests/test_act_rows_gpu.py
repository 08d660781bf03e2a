"""The per-token activation quantizer at the edges of its row mapping, by the checks of test_kernels_gpu:
one row, rows per CTA that cross the eight whose states are formed together, rows of each thread count
and length class (registers, shared memory, 512 threads with LET sums), ragged last vectors; and rows
and divisors that leave the range of the fast exact division."""
import pytest
import torch

import test_block_gpu as B
import test_kernels_gpu as K
from _stagewise import compare_step
from paper_2308_13137_gb300 import _lib
from paper_2308_13137_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T,C,nbits,let", [
    (1, 512, 4, True),
    (2800, 264, 4, True),        # ten rows a CTA: a second set of states
    (700, 5120, 4, True),        # 512 threads
    (40, 9000, 6, True),
    (30, 13000, 4, True),
    (33, 28672, 4, False),       # through shared memory, 512 threads
    (9, 4104, 3, False),
    (5, 12288, 4, True),         # the row alone takes the 48 KB a CTA has without asking for more
    (9, 16384, 4, True),
    (11, 16392, 4, True),        # the longest form of the LET column sums
    (310, 20488, 6, True),       # two rows a CTA and more
    (7, 28672, 4, True),
    (640, 4096, 4, False),
])
def test_act_row_edges(cuda_lib, T, C, nbits, let):
    K.test_act_quant_fwd_bwd(cuda_lib, T, C, nbits, let)


@pytest.mark.parametrize("C", [1024, 6144])
def test_division_ranges(cuda_lib, C):
    """Zeros, numerators below 2^-60 and divisors beyond 2^40: the quantizer input is the IEEE quotient either
    way, so the codes, h and z are those of the same row divided beforehand (LET off)."""
    T = 12
    g = torch.Generator().manual_seed(C)
    X, s, d = torch.randn(T, C, generator=g), torch.exp(0.3 * torch.randn(C, generator=g)), torch.zeros(C)
    X[1] = 0
    X[2, ::7] = 0
    X[3] *= 2.0 ** -70
    X[4, 5] = 2.0 ** 50
    X[5, ::3] *= 2.0 ** -66
    s[17] = 2.0 ** 45
    s[C - 1] = 2.0 ** -45
    X[:, C - 1] *= 2.0 ** -45
    Xt = X / s                                    # IEEE single precision, one rounding
    out = []
    for x, sv, dv in ((X, s, d), (Xt, None, None)):
        dev = lambda v: None if v is None else v.cuda().contiguous()
        e = lambda *sh, dt=torch.float32: torch.empty(*sh, dtype=dt, device="cuda")
        Xq, h, z = e(T, C, dt=torch.bfloat16), e(T), e(T, dt=torch.int32)
        i0, i1 = e(T, dt=torch.int32), e(T, dt=torch.int32)
        _lib.omq_act_quant_per_token(T, C, dev(x), dev(sv), dev(dv), Xq, None, h, z, i0, i1, _lib.make_cfg(abits=4))
        out.append([v.cpu() for v in (Xq, h, z, i0, i1)])
    for a, b in zip(*out):
        assert torch.equal(a, b)


@pytest.mark.parametrize("T,ffn", [(1, 512), (70, 1032), (33, 11008), (9, 28672)])
def test_swiglu_rows(cuda_lib, T, ffn):
    """The SwiGLU rows of the block (one loop for every length), stage by stage against the oracle."""
    shape = I.BlockShape(f"swiglu_{T}_{ffn}", T=T, d=256, n_heads=2, n_kv=1, ffn=ffn, wbits=4, abits=4, group=0, let=1)
    _, got = B._run(shape)
    W, x, th, yfp = got["inputs"]
    compare_step(shape, W, x, th, yfp, got["y"], got["loss"], {k: v for k, v in got.items() if k.startswith("d")},
                 got["saved"], shape.name)


@pytest.mark.parametrize("T,d", [(33, 4104), (21, 8192), (9, 8200), (5, 16392)])
def test_long_rmsnorm_rows(cuda_lib, T, d):
    """RMSNorm rows of 512 and 1024 threads, of four and eight vectors each, in a block checked stage by stage."""
    shape = I.BlockShape(f"rms_{T}_{d}", T=T, d=d, n_heads=1, n_kv=1, ffn=128, wbits=4, abits=4, group=0,
                         let=int(d <= 16384))
    _, got = B._run(shape)
    W, x, th, yfp = got["inputs"]
    compare_step(shape, W, x, th, yfp, got["y"], got["loss"], {k: v for k, v in got.items() if k.startswith("d")},
                 got["saved"], shape.name)


@pytest.mark.parametrize("T,d", [(5, 16392), (3, 20480)])
def test_longest_rmsnorm_rows_with_let(cuda_lib, T, d):
    """RMSNorm rows past 16 K columns with LET: the column sums' longest form, whose second pass reads the row again."""
    shape = I.BlockShape(f"rms_let_{T}_{d}", T=T, d=d, n_heads=1, n_kv=1, ffn=128, wbits=4, abits=4, group=0, let=1)
    _, got = B._run(shape)
    W, x, th, yfp = got["inputs"]
    compare_step(shape, W, x, th, yfp, got["y"], got["loss"], {k: v for k, v in got.items() if k.startswith("d")},
                 got["saved"], shape.name)
