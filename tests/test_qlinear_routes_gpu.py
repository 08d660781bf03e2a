"""omq_qlinear_bwd against the composition of the kernel-level entry points it stands for (the stored
product dW_hat = dY^T X_hat, then omq_lwc_fakequant_bwd; dX_hat = dY W_hat, then
omq_act_quant_per_token_bwd), at ragged token counts and at the sizes where its LWC backward moves
between the product's epilogue and the separate pass.  Both sides multiply the same bf16 operands and
add in fp32, in another order: 2e-5 relative (sums of up to 1.5e5 terms; ddelta, a difference of two
such sums, against the larger of them)."""
import pytest
import torch

from paper_2308_13137_gb300 import _lib

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T,Cin,Cout,abits,group,let", [
    (1, 64, 8, 16, 0, 0),            # one token, one column of tiles
    (129, 512, 264, 4, 0, 1),        # one row past a slab of the column sums
    (300, 520, 136, 8, 0, 1),        # Cin not a multiple of the epilogue's 32-column chunk
    (260, 768, 512, 16, 128, 0),
    (127, 384, 200, 4, 64, 0),
    (200, 512, 256, 4, 128, 1),      # LET with groups: the separate pass
    (1031, 1024, 1000, 4, 0, 1),
])
def test_qlinear_bwd_routes(cuda_lib, T, Cin, Cout, abits, group, let, flat=False):
    g = torch.Generator().manual_seed(T + Cin + Cout)
    dev = lambda t: t.cuda().contiguous()
    n = lambda *s: torch.randn(*s, generator=g)
    e = lambda *s, dt=torch.float32: torch.empty(*s, dtype=dt, device="cuda")
    ng = Cin // (group or Cin)
    X, W, dY = dev(n(T, Cin)), dev((0.02 * n(Cout, Cin)).to(torch.bfloat16)), dev(n(T, Cout) / T)
    gl, bl = dev(4 + n(Cout, ng)), dev(4 + n(Cout, ng))
    s, d = (dev(torch.exp(0.2 * n(Cin))), dev(0.1 * n(Cin))) if let else (None, None)
    if flat:
        if let:
            s = dev(torch.exp2(torch.randint(-2, 3, (Cin,), generator=g).float()))
        W[::3] = (64.0 / s).to(torch.bfloat16) if let else 64.0
        gl, bl = dev(4 + 0 * gl), dev(4 + 0 * bl)
    cfg = _lib.make_cfg(4, abits, group, let)
    kinds = [torch.bfloat16] + [torch.float32] + 3 * [torch.int32] + [torch.bfloat16] + [torch.float32] + \
        3 * [torch.int32] + [torch.float32]
    keep = [e(k, dt=t) for k, t in zip(_lib.omq_qlinear_saved_sizes(T, Cin, Cout, cfg), kinds)]
    saved = _lib.omq_qlinear_saved(*[t.data_ptr() for t in keep])
    Y = e(T, Cout)
    _lib.omq_qlinear_fwd(T, Cin, Cout, X, W, None, s, d, gl, bl, Y, saved, cfg)
    ws = torch.empty(_lib.omq_qlinear_workspace_size(T, Cin, Cout, cfg), dtype=torch.uint8, device="cuda")
    dX, dg, db, ds, dd = e(T, Cin), e(Cout, ng), e(Cout, ng), e(Cin) if let else None, e(Cin) if let else None
    _lib.omq_qlinear_bwd(T, Cin, Cout, X, W, s, d, gl, bl, saved, dY, dX, dg, db, ds, dd, ws, cfg)

    w_hat, h, z, iM, im, x_hat, ha, za, iMa, ima, _ = keep
    dYb = dY.to(torch.bfloat16)
    dW, dXh = e(Cout, Cin), e(T, Cin)
    _lib.omq_gemm_bf16(Cout, Cin, T, 1, dYb, Cout, 0, 0, x_hat, Cin, 0, 0, dW, None, Cin, 0)
    _lib.omq_gemm_bf16(T, Cin, Cout, 1, dYb, Cout, 0, 1, w_hat, Cin, 0, 0, dXh, None, Cin, 0)
    rg, rb, rX = e(Cout, ng), e(Cout, ng), e(T, Cin)
    rs, rd = (e(Cin), e(Cin)) if let else (None, None)
    ws1 = torch.empty(_lib.omq_lwc_bwd_workspace_size(Cout, Cin), dtype=torch.uint8, device="cuda")
    dB = dY.double().sum(0).float() if let else None
    _lib.omq_lwc_fakequant_bwd(Cout, Cin, W, s, None, gl, bl, h, z, iM, im, dW, rg, rb, None, rs, None, dB, rd, ws1, cfg)
    lwc_dd = rd.clone() if let else None
    ws2 = torch.empty(_lib.omq_act_bwd_workspace_size(T, Cin), dtype=torch.uint8, device="cuda")
    acc = _lib.make_cfg(4, abits, group, let, accumulate=1)
    st = (ha, za, iMa, ima) if abits < 16 else (None,) * 4
    _lib.omq_act_quant_per_token_bwd(T, Cin, X, s, d, *st, dXh, rX, rs, rd, ws2, acc)
    torch.cuda.synchronize()
    rel = lambda a, b, by=None: float((a.double() - b.double()).norm() / (b if by is None else by).double().norm())
    assert rel(dg, rg) < 2e-5 and rel(db, rb) < 2e-5 and rel(dX, rX) < 2e-5
    if let:
        assert rel(ds, rs) < 2e-5
        assert rel(dd, rd, lwc_dd) < 2e-5


@pytest.mark.parametrize("T,Cin,Cout,abits,group,let", [
    (260, 768, 512, 16, 128, 0),
    (130, 512, 256, 16, 0, 0),
    (130, 512, 256, 4, 0, 1),
])
def test_flat_rows(cuda_lib, T, Cin, Cout, abits, group, let):
    """Every third row equal to 64 in the quantizer's input: its step is the floor, 1e-5, and its quotients, 6.4e6,
    are past the range of the fast rounding, next to rows that are inside."""
    test_qlinear_bwd_routes(cuda_lib, T, Cin, Cout, abits, group, let, flat=True)


@pytest.mark.parametrize("T,Cin,Cout,group,let,tile", [
    (130, 512, 120, 0, 1, (64, 1)),
    (300, 768, 512, 32, 0, (64, 1)),
    (1031, 1032, 1032, 0, 1, (128, 1)),      # ragged last tile and last chunk
    (1031, 512, 3080, 0, 0, (128, 1)),
    (260, 768, 512, 64, 0, (128, 1)),
    (260, 768, 120, 128, 0, (256, 1)),
    (260, 768, 512, 128, 0, (256, 2)),
    (1531, 4104, 2048, 0, 1, (256, 2)),
    (1531, 4096, 2048, 0, 0, (256, 2)),
    (200, 512, 256, 128, 1, (0, 0)),         # LET with groups, groups of 16: the separate pass
    (200, 512, 256, 16, 0, (0, 0)),
])
def test_lwc_epilogue_tiles(cuda_lib, T, Cin, Cout, group, let, tile):
    """Every output tile of the weight-gradient product with the LWC epilogue, and the pass where it has none."""
    if not (group and let):
        assert _lib.omq_gemm_tile(Cout, Cin, T, group or Cin) == tile
    test_qlinear_bwd_routes(cuda_lib, T, Cin, Cout, 4, group, let)
