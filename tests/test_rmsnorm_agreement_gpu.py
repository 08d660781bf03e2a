"""Forward and backward of the first RMSNorm form the same quantizer input.  Every token is the same row of integers, so
that its sum of squares is exact, and delta_1 is the rounded product x * rstd: the input (x * rstd - delta_1) / s_1
is exactly zero.  A backward that joined the product with the subtraction would find the product's rounding
error there instead, and ds_1 = -sum_t dX~ X~ / s_1, whose weight part is zero with the quantized input, would not be
zero."""
import numpy as np
import pytest
import torch

from paper_2308_13137_gb300 import inputs as I
from paper_2308_13137_gb300.block import BlockState

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d", [256, 8192])
def test_rmsnorm_input_agrees(cuda_lib, d):
    shape = I.BlockShape(f"agree_{d}", T=16, d=d, n_heads=2, n_kv=2, ffn=384, wbits=4, abits=4, group=0, let=1)
    W = I.make_block_weights(shape, seed=3)
    th = I.make_block_theta(shape, W, I.make_block_input(shape, sample=0, weight_seed=3), seed=4, perturb=True)
    top = int(np.sqrt((2 ** 24 - 1) / d))
    row = np.random.default_rng(d).integers(1, top + 1, d).astype(np.float32) * np.where(np.arange(d) % 3, 1, -1)
    row = row.astype(np.float32)
    ms = np.float32(np.float32(np.square(row.astype(np.float64)).sum()) / np.float32(d))
    rstd = np.float32(1) / np.sqrt(ms + np.float32(shape.rms_eps))
    th["d1"] = (row * rstd).astype(np.float32)
    th["s1"] = np.full(d, 2.0 ** -6, np.float32)
    x = np.tile(row, (shape.T, 1))
    st = BlockState(shape, W, th)
    xd = torch.from_numpy(x).cuda()
    st.step(xd, xd + torch.randn(shape.T, d, generator=torch.Generator().manual_seed(1)).cuda())
    torch.cuda.synchronize()
    g = st.split_grads()
    assert int(st.status.item()) == 0
    assert float(np.abs(g["dd1"]).max()) > 0
    assert float(np.abs(g["ds1"]).max()) == 0
