"""Rows and groups of NaN alone: no element equals their extreme, and the forward saves one of their columns as the index
of the max and of the min, which the backward reads and writes at.  Every forward form, then one block step, which
returns a NaN loss and leaves the GPU usable."""
import numpy as np
import pytest
import torch

from paper_2308_13137_gb300 import _lib
from paper_2308_13137_gb300 import inputs as I
from paper_2308_13137_gb300.block import BlockState

pytestmark = pytest.mark.gpu

NAN = float("nan")


def _i32(*s):
    return torch.full(s, -1, dtype=torch.int32, device="cuda")


@pytest.mark.parametrize("C", [8, 1024, 4096, 6144, 12288, 32768])     # register and shared-memory rows
@pytest.mark.parametrize("let", [False, True])
def test_act_rows(cuda_lib, C, let):
    T = 5
    X = torch.randn(T, C, generator=torch.Generator().manual_seed(C)).cuda()
    X[1], X[3, 1:] = NAN, NAN                     # a whole row, and all but its first column
    X[4, :-1] = NAN
    s, d = (torch.ones(C, device="cuda"), torch.zeros(C, device="cuda")) if let else (None, None)
    Xq, h, z, a, b = torch.empty(T, C, device="cuda", dtype=torch.bfloat16), torch.empty(T, device="cuda"), _i32(T), _i32(T), _i32(T)
    _lib.omq_act_quant_per_token(T, C, X, s, d, Xq, None, h, z, a, b, _lib.make_cfg(abits=4, let=let))
    for i in (a.tolist(), b.tolist()):
        assert i[1] == 0 and i[3] == 0 and i[4] == C - 1
        assert all(0 <= v < C for v in i)


@pytest.mark.parametrize("Cin,group", [
    (512, 8), (512, 16), (512, 32), (512, 64), (512, 128), (512, 256),       # lane segments; the grouped kernel
    (512, 0), (12288, 0), (20000, 0), (40960, 0),                            # one group a row, every row form
])
@pytest.mark.parametrize("scaled", [False, True])
def test_lwc_groups(cuda_lib, Cin, group, scaled):
    Cout, g = 9, group or Cin
    ng = Cin // g
    W = torch.randn(Cout, Cin, generator=torch.Generator().manual_seed(Cin)).to(torch.bfloat16).cuda()
    W[4, Cin - g:] = NAN                          # the last group of a row
    W[7] = NAN
    W[2, :g - 1] = NAN
    s = torch.ones(Cin, device="cuda") if scaled else None
    lg = torch.full((Cout, ng), 4.0, device="cuda")
    Wq, h, z, a, b = torch.empty_like(W), torch.empty(Cout, ng, device="cuda"), _i32(Cout, ng), _i32(Cout, ng), _i32(Cout, ng)
    _lib.omq_lwc_fakequant_fwd(Cout, Cin, W, s, None, lg, lg, Wq, None, h, z, a, b, None, None, None,
                               _lib.make_cfg(wbits=4, group=group))
    first = (torch.arange(ng) * g).int()
    for i in (a.cpu(), b.cpu()):
        assert bool(((i >= first) & (i < first + g)).all())
        assert int(i[2, 0]) == g - 1


@pytest.mark.parametrize("group,let", [(0, 1), (128, 0)])
def test_block_step(cuda_lib, group, let):
    shape = I.BlockShape(f"nan_{group}", T=40, d=256, n_heads=2, n_kv=1, ffn=384, wbits=4, abits=4, group=group, let=let)
    W = I.make_block_weights(shape, seed=3)
    x = I.make_block_input(shape, sample=0, weight_seed=3)
    st = BlockState(shape, W, I.make_block_theta(shape, W, x, seed=4, perturb=True))
    yfp = torch.from_numpy(x).cuda()
    good = torch.from_numpy(x).cuda()
    ref = float(st.step(good, yfp).item())
    bad = x.copy()
    bad[11, 5] = np.nan                           # one value: its RMSNorm makes the token NaN
    assert np.isnan(float(st.step(torch.from_numpy(bad).cuda(), yfp).item()))
    assert float(st.step(good, yfp).item()) == ref and np.isfinite(ref)
    assert int(st.status.item()) == 0
