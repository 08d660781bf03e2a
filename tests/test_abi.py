"""Host-side checks of the C ABI that need no GPU: the library loads, exports every function
include/omq.h declares, sizes its workspaces, and rejects bad arguments before any launch."""
import ctypes
import os

import pytest

from paper_2308_13137_gb300 import _lib, inputs as I

pytestmark = pytest.mark.skipif(not os.path.exists(_lib.LIB_PATH), reason="libomq.so not built")


def test_exports_every_declared_function():
    L = _lib.lib()
    names = _lib.header_functions()
    assert len(names) >= 15
    for n in names:
        assert hasattr(L, n), n
        assert n in _lib._SIGS, f"binding lacks {n}"
    assert _lib.omq_version() == 1
    assert _lib.omq_status_string(3).startswith("misaligned")


def test_every_exported_function_is_declared():
    """The reverse direction: no omq_ symbol leaves the library undocumented by the header."""
    import shutil
    import subprocess
    if not shutil.which("nm"):
        pytest.skip("nm not available")
    out = subprocess.run(["nm", "-D", "--defined-only", _lib.LIB_PATH], capture_output=True, text=True,
                         check=True).stdout
    exported = {f[2] for f in (line.split() for line in out.splitlines())
                if len(f) == 3 and f[1] == "T" and f[2].startswith("omq_")}
    assert exported and exported <= set(_lib.header_functions()), sorted(exported - set(_lib.header_functions()))


def _cfg(**kw):
    base = dict(wbits=4, abits=16, group=128, let=0, h_eps=1e-5, accumulate=0, dev_status=None, pbits=0, wprep=0)
    base.update(kw)
    return _lib.omq_qcfg(base["wbits"], base["abits"], base["group"], base["let"], base["h_eps"],
                         base["accumulate"], base["dev_status"], base["pbits"], base["wprep"])


FAKE = 0x10000     # 16-byte aligned dummy address: every call below returns before touching it


def _lwc_fwd(Cout, Cin, cfg, W=FAKE, Wq=FAKE):
    L = _lib.lib()
    return L.omq_lwc_fakequant_fwd(None, Cout, Cin, W, None, None, FAKE, FAKE, Wq, None, FAKE, FAKE, FAKE, FAKE,
                                   None, None, None, ctypes.byref(cfg) if cfg is not None else None)


def test_argument_errors_before_launch():
    assert _lwc_fwd(0, 512, _cfg()) == 2                       # OMQ_ERR_SHAPE
    assert _lwc_fwd(64, 500, _cfg(group=0)) == 3               # inner dimension not a multiple of 8
    assert _lwc_fwd(64, 512, _cfg(group=96)) == 2              # group does not divide Cin
    assert _lwc_fwd(64, 512, _cfg(wbits=1)) == 4               # OMQ_ERR_UNSUPPORTED
    assert _lwc_fwd(64, 512, _cfg(wbits=12)) == 4
    assert _lwc_fwd(64, 512, None) == 1                        # OMQ_ERR_INVALID_ARG
    assert _lwc_fwd(64, 512, _cfg(wprep=2)) == 1               # operand preparation mode outside {0, 1}
    assert _lwc_fwd(64, 512, _cfg(), W=FAKE + 4) == 3          # misaligned pointer
    L = _lib.lib()
    # workspace too small
    assert L.omq_block_loss(None, 1024, FAKE, FAKE, FAKE, None, None, FAKE, 4) == 7
    # GEMM: misaligned leading dimension
    assert L.omq_gemm_bf16(None, 128, 128, 64, 1, FAKE, 60, 0, 1, FAKE, 64, 0, 1, FAKE, None, 128, 0, 1.0,
                           None, None, 0, 0.0, 0, None) == 3
    # GEMM: bad causal mode
    assert L.omq_gemm_bf16(None, 128, 128, 64, 1, FAKE, 64, 0, 1, FAKE, 64, 0, 1, FAKE, None, 128, 0, 1.0,
                           None, None, 0, 0.0, 7, None) == 1


def test_softmax_quant_argument_errors():
    """The softmax-output quantizer's bit width and step floor are checked before any launch."""
    L = _lib.lib()
    assert _lwc_fwd(64, 512, _cfg(pbits=9)) == 4               # pbits outside 2..8 (0 / 16 = off)
    assert _lwc_fwd(64, 512, _cfg(pbits=1)) == 4
    for bits in (1, 9, 16, 0):
        assert L.omq_attention_pq_fwd(None, 256, 2, 2, FAKE, 256, FAKE, FAKE, 256, FAKE, 256, FAKE, bits, 1e-5,
                                      FAKE, None) == 4
        assert L.omq_attention_pq_bwd(None, 256, 2, 2, FAKE, 256, FAKE, FAKE, 256, FAKE, FAKE, 256, FAKE, 256, FAKE,
                                      FAKE, 256, bits, FAKE, FAKE, None) == 4
    assert L.omq_attention_pq_fwd(None, 256, 2, 2, FAKE, 256, FAKE, FAKE, 256, FAKE, 256, FAKE, 8, 0.0,
                                  FAKE, None) == 1             # h_eps must be positive
    assert L.omq_attention_pq_fwd(None, 256, 2, 2, FAKE, 256, FAKE, FAKE, 256, FAKE, 256, FAKE, 8, 1e-5,
                                  None, None) == 1             # the row records are required


def test_qlinear_saved_sizes():
    """Element counts of the single linear's saved arrays, in the struct's field order."""
    n = _lib.omq_qlinear_saved_sizes(256, 512, 384, _cfg(group=128))
    ng = 384 * 4
    assert n == [384 * 512, ng, ng, ng, ng, 256 * 512, 256, 256, 256, 256, 384]
    assert _lib.omq_qlinear_saved_sizes(256, 512, 384, _cfg(group=0))[1] == 384
    with pytest.raises(_lib.OmqError):
        _lib.omq_qlinear_saved_sizes(256, 512, 384, _cfg(group=96))       # 96 does not divide 512


def test_block_workspace_sizes():
    sh = I.SHAPES["llama7b_w4a4"]
    s = _lib.omq_block_shape(sh.T, sh.d, sh.n_heads, sh.n_kv, sh.head_dim, sh.ffn, sh.rms_eps, sh.rope_theta)
    ws = _lib.omq_block_workspace_size(s, _cfg(wbits=4, abits=4, group=0, let=1))
    assert 2e9 < ws < 8e9                                      # a few GB for the 7B block step
    bad = _lib.omq_block_shape(sh.T, sh.d, 32, 5, 128, sh.ffn, 1e-6, 1e4)    # heads not divisible
    assert _lib.omq_block_workspace_size(bad, _cfg()) == 0
    hd64 = _lib.omq_block_shape(sh.T, sh.d, 64, 64, 64, sh.ffn, 1e-6, 1e4)   # head_dim must be 128
    assert _lib.omq_block_workspace_size(hd64, _cfg()) == 0
    assert _lib.omq_qlinear_workspace_size(256, 512, 512, _cfg()) > 512 * 512 * 4
    # the softmax-quantized step carries two small per-row arrays more
    ws8 = _lib.omq_block_workspace_size(s, _cfg(wbits=4, abits=4, group=0, let=1, pbits=8))
    assert ws < ws8 < ws + 16 * sh.n_heads * sh.T * 4
    assert _lib.omq_block_workspace_size(s, _cfg(wbits=4, abits=4, group=0, let=1, pbits=12)) == 0


def _refused(fn, args, at, off, code=3):
    """fn with args is refused with `code` when the pointer at position `at` is moved by `off` bytes."""
    a = list(args)
    a[at] = FAKE + off
    return fn(*a) == code


def test_vector_pointers_must_be_aligned():
    """Pointers that the kernels read or write in 16-byte vectors are refused on the host when they are not 16-byte
    aligned."""
    L = _lib.lib()
    c = ctypes.byref(_cfg(abits=4, group=0, let=1))
    act_f = [None, 4, 512, FAKE, FAKE, FAKE, FAKE, FAKE, FAKE, FAKE, FAKE, FAKE, c]
    for i in (3, 4, 5, 6):                                   # X, s, delta, Xq
        assert _refused(L.omq_act_quant_per_token, act_f, i, 4)
    assert _refused(L.omq_act_quant_per_token, act_f, 7, 2)  # codes, written four at a time
    act_b = [None, 4, 512, FAKE, FAKE, FAKE, FAKE, FAKE, FAKE, FAKE, FAKE, FAKE, FAKE, FAKE, FAKE, 1 << 30, c]
    for i in (3, 4, 5, 10, 11, 14):                          # X, s, delta, dXq, dX, workspace
        assert _refused(L.omq_act_quant_per_token_bwd, act_b, i, 8)
    lwc_f = [None, 64, 512, FAKE, FAKE, None, FAKE, FAKE, FAKE, None, FAKE, FAKE, FAKE, FAKE, FAKE, None, FAKE, c]
    for i in (3, 4, 8, 14):                                  # W, s, Wq, bias_delta
        assert _refused(L.omq_lwc_fakequant_fwd, lwc_f, i, 8)
    sv = _lib.omq_qlinear_saved(*[FAKE] * 11)
    ql_f = [None, 4, 512, 64, FAKE, FAKE, FAKE, FAKE, FAKE, FAKE, FAKE, FAKE, ctypes.byref(sv), c]
    for i in (4, 5, 7, 8, 11):                               # X, W, s, delta, Y
        assert _refused(L.omq_qlinear_fwd, ql_f, i, 8)
    ql_b = [None, 4, 512, 64, FAKE, FAKE, FAKE, FAKE, FAKE, FAKE, ctypes.byref(sv), FAKE, FAKE, FAKE, FAKE, FAKE, FAKE, FAKE,
            1 << 30, c]
    for i in (4, 5, 6, 7, 11, 12, 17):                       # X, W, s, delta, dY, dX, workspace
        assert _refused(L.omq_qlinear_bwd, ql_b, i, 8)


def test_let_vectors_must_be_aligned():
    """The block's LET vectors: all of them with a kv head per query head; with shared kv heads so and do are
    expanded to copies first, so theirs does not matter."""
    L, c = _lib.lib(), ctypes.byref(_cfg(abits=4, group=0, let=1))
    w = _lib.omq_block_weights(FAKE, FAKE, FAKE, FAKE)
    for n_kv, names in ((2, ["s1", "d1", "so", "do_", "sa", "s2", "d2"]), (1, ["s1", "d1", "sa", "s2", "d2"])):
        s = _lib.omq_block_shape(16, 256, 2, n_kv, 128, 384, 1e-6, 1e4)
        for n in names + [None]:
            th = _lib.omq_block_params(*[FAKE] * len(_lib.PARAM_FIELDS))
            if n:
                setattr(th, n, FAKE + 8)
            e = L.omq_block_forward(None, ctypes.byref(s), ctypes.byref(w), ctypes.byref(th), FAKE, FAKE, FAKE, 0, c)
            assert e == (3 if n else 7), (n_kv, n, e)        # OMQ_ERR_ALIGN, or the workspace of no bytes


def test_qlinear_workspace_of_bad_shapes():
    """A shape without tokens or columns has no workspace, whatever the group (a query in a process of its own: it
    used to end the process)."""
    import subprocess
    import sys
    code = ("import ctypes, sys; sys.path.insert(0, %r); from paper_2308_13137_gb300 import _lib; L = _lib.lib()\n"
            "for g in (0, 128):\n"
            "    c = _lib.make_cfg(4, 16, g, 0)\n"
            "    for s in ((4, 0, 64), (4, 512, 0), (0, 512, 64), (-1, 512, 64), (4, -512, 64)):\n"
            "        for p in (ctypes.byref(c), None):\n"
            "            assert L.omq_qlinear_workspace_size(*s, p) == 0, (s, g)\n")
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", code % root], capture_output=True, text=True)
    assert r.returncode == 0, (r.returncode, r.stderr)


def test_qlinear_workspace_serves_every_configuration():
    """One size per shape, whatever the group and the LET setting: a buffer sized once is accepted with any of them."""
    L = _lib.lib()
    for T, Cin, Cout in ((256, 512, 512), (1, 8, 8), (300, 520, 136), (2048, 4096, 11008)):
        sizes = {L.omq_qlinear_workspace_size(T, Cin, Cout, ctypes.byref(_cfg(group=g, let=let)))
                 for g in (0, 8, 32, 64, 128, 256) for let in (0, 1)}
        sizes.add(L.omq_qlinear_workspace_size(T, Cin, Cout, None))
        assert len(sizes) == 1 and sizes.pop() > 2 * T * Cout + 4 * Cout * Cin + 4 * T * Cin


def test_gemm_tile_query():
    assert _lib.omq_gemm_tile(100, 8, 8) == (64, 1)
    assert _lib.omq_gemm_tile(2048, 4096, 4096) == (256, 2)
    assert _lib.omq_gemm_tile(512, 512, 256, 16) == (0, 0)        # the epilogue takes groups of 32 and more
    for bad in ((0, 8, 8, 0), (8, 8, 0, 0), (8, 512, 8, 96), (8, 8, 8, -1)):
        with pytest.raises(_lib.OmqError):
            _lib.omq_gemm_tile(*bad)
