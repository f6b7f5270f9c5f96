"""Bit-exact parity of every CUDA entry point with the CPU oracle, element by element, on seeded
inputs that span several tiles plus ragged tails, and on the edge cases of each operator.
The whole path is integer, so the tolerance is zero everywhere."""
import ctypes
import os
import time

import numpy as np
import pytest

from paper_2607_24981_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

TENSOR_MEMORY = not os.environ.get("ILWDETR_ATTENTION_TC", "").startswith("0")


@pytest.fixture(scope="module")
def ilw():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2607_24981_gb300 as m
    from paper_2607_24981_gb300 import build

    build.build()
    m.lib()
    return m


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def host(t):
    torch.cuda.synchronize()
    return t.cpu().numpy()


def assert_same(got, want, what=""):
    got = np.asarray(got)
    want = np.asarray(want).astype(got.dtype)
    if not np.array_equal(got, want):
        bad = np.argwhere(got != want)
        i = tuple(bad[0])
        raise AssertionError(f"{what}: {len(bad)} mismatches, first at {i}: gpu={got[i]} oracle={want[i]}")


# ------------------------------------------------------------------------------ GEMM
@pytest.mark.parametrize("M,N,K", [(1, 1, 16), (37, 29, 64), (130, 200, 384), (257, 129, 80),
                                   (300, 1152, 384), (128, 384, 1536)])
@pytest.mark.parametrize("out_bits,mode", [(8, "calibrated"), (8, "literal"), (16, "calibrated"), (32, "literal"),
                                           (108, "calibrated")])
def test_gemm_requant(ilw, orc, M, N, K, out_bits, mode):
    """out_bits 108 (ILW_I8_IN_F16): the out_bits 8 result carried as float16."""
    A = synth.uniform_int(1, f"A{M}{K}", (M, K), -127, 127, np.int8)
    W, b, m, s = synth.gemm_params(1, f"W{N}{K}", N, K, 73.0, 40.0, mode)
    Wp = ilw.pack_weight(dev(W))
    got = ilw.gemm_requant(dev(A), Wp, N, dev(b), dev(m), dev(s), out_bits)
    want = orc.gemm_requant(A, W, b, m, s, 8 if out_bits == ilw.I8_IN_F16 else out_bits)
    if out_bits == ilw.I8_IN_F16:
        assert got.dtype == torch.float16
    assert_same(host(got), want, "gemm")


def test_gemm_extremes_and_residual(ilw, orc):
    """All-(+127) and all-(-127) operands reach the largest accumulators; the residual term
    broadcasts rows (row % rows) as the patch embedding's position term does."""
    M, N, K = 200, 96, 1536
    A = np.full((M, K), 127, np.int8)
    A[::2] = -127
    W = np.full((N, K), 127, np.int8)
    W[:, ::3] = -127
    _, b, m, s = synth.gemm_params(2, "Wx", N, K, 73.0, 40.0, "literal")
    res = synth.uniform_int(2, "res", (50, N), -32767, 32767, np.int16)
    Wp = ilw.pack_weight(dev(W))
    got = ilw.gemm_requant(dev(A), Wp, N, dev(b), dev(m), dev(s), 16, res=dev(res), m_r=3 << 29, s_r=31)
    want = orc.gemm_requant(A, W, b, m, s, 16, res, 3 << 29, 31)
    assert_same(host(got), want, "gemm+res")
    got32 = ilw.gemm_requant(dev(A), Wp, N, dev(b), None, None, 32)
    assert_same(host(got32), orc.gemm_requant(A, W, b, m, s, 32), "gemm raw")


@pytest.mark.parametrize("M,N,K,I0", [(100, 96, 64, 300), (513, 768, 192, 1 << 10), (64, 1536, 384, 2047)])
def test_gemm_gelu(ilw, orc, M, N, K, I0):
    A = synth.uniform_int(3, "Ag", (M, K), -127, 127, np.int8)
    W, b, m, s = synth.gemm_params(3, "Wg", N, K, 73.0, 2.0 * I0, "calibrated")
    Wp = ilw.pack_weight(dev(W))
    m_g, s_g = 3 << 29, 40
    got = ilw.gemm_gelu(dev(A), Wp, N, dev(b), dev(m), dev(s), {"I0": I0}, m_g, s_g)
    g = orc.gemm_requant(A, W, b, m, s, 16)
    gi = orc.sdshiftgelu(g, I0).astype(np.int64)
    want = np.array([[orc.sat(orc.rq(int(v), m_g, s_g), 8) for v in row] for row in gi], np.int8)
    assert_same(host(got), want, "gemm_gelu")


# fp16-carried int8 A (ilwdetr_gemm a_form ILW_I8_IN_F16): resident-weight tiles of 192 (N % 192 == 0)
# and 128 columns, streamed weights for K > 1024, ragged M / N, every epilogue form
@pytest.mark.parametrize("M,N,K", [(1, 1, 16), (37, 29, 64), (300, 1152, 384), (257, 384, 1024), (130, 200, 384),
                                   (128, 96, 256), (12800, 1536, 384), (333, 384, 1536), (64, 192, 1040)])
@pytest.mark.parametrize("kind", ["rq8", "rq16res", "f16", "raw32", "gelu8", "gelu_f16"])
def test_gemm_f16_operand(ilw, orc, M, N, K, kind):
    if M * N * K > 1e9 and kind not in ("f16", "gelu_f16", "rq16res"):
        pytest.skip("the large case runs the encoder's forms only")
    A = synth.uniform_int(11, f"Af{M}{K}", (M, K), -127, 127, np.int8)
    I0 = 700
    W, b, m, s = synth.gemm_params(11, f"Wf{N}{K}", N, K, 73.0, 2.0 * I0 if kind.startswith("gelu") else 40.0)
    Wp = ilw.pack_weight(dev(W))
    Ad = dev(A.astype(np.float16))
    F16 = ilw.I8_IN_F16
    if kind.startswith("gelu"):
        m_g, s_g = 3 << 29, 40
        got = ilw.gemm(Ad, Wp, N, dev(b), dev(m), dev(s), F16 if kind == "gelu_f16" else 8, gelu={"I0": I0},
                       m_g=m_g, s_g=s_g)
        gi = orc.sdshiftgelu(orc.gemm_requant(A, W, b, m, s, 16), I0).astype(np.int64)
        want = np.array([[orc.sat(orc.rq(int(v), m_g, s_g), 8) for v in row] for row in gi], np.int8) \
            if M * N <= 1 << 20 else orc.requant(gi.astype(np.int32), m_g, s_g, out_bits=8)
    elif kind == "rq16res":
        res = synth.uniform_int(12, "resf", (M, N), -32767, 32767, np.int16)
        got = ilw.gemm(Ad, Wp, N, dev(b), dev(m), dev(s), 16, res=dev(res), m_r=3 << 29, s_r=31)
        want = orc.gemm_requant(A, W, b, m, s, 16, res, 3 << 29, 31)
    else:
        ob = {"rq8": 8, "f16": F16, "raw32": 32}[kind]
        got = ilw.gemm(Ad, Wp, N, dev(b), dev(m), dev(s), ob)
        want = orc.gemm_requant(A, W, b, m, s, 8 if ob == F16 else ob)
    if kind in ("f16", "gelu_f16"):
        assert got.dtype == torch.float16
    assert_same(host(got), want, f"gemm fp16-A {kind}")


# ------------------------------------------------------------------------------ Shiftmax rows
@pytest.mark.parametrize("L", [1, 3, 4, 63, 64, 65, 128, 400, 1600, 1664, 2048, 2100])
def test_shiftmax_rows(ilw, orc, L):
    rows = 257
    X = synth.uniform_int(4, f"smx{L}", (rows, L), -(1 << 15), 1 << 15)
    for I0, sd in ((1 << 11, -1), (1 << 13, -1), (3000, 0), (5000, 7)):
        got = ilw.shiftmax_rows(dev(X), {"I0": I0, "s_d": sd})
        P, *_ = orc.shiftmax_rows(X, I0, s_d=sd)
        assert_same(host(got), P, f"shiftmax L={L} I0={I0} s_d={sd}")


def test_shiftmax_rows_edge_values(ilw, orc):
    """Full-int32 scores (differences far below the ShiftExp clamp), constant rows, a strided
    (non-contiguous) layout and the largest I0."""
    X = synth.uniform_int(5, "smxe", (64, 100), -(1 << 31), (1 << 31) - 1)
    X[3] = 7
    X[4, ::2] = 2**31 - 1
    X[4, 1::2] = -(2**31)
    for I0 in (1, 2, (1 << 15) - 1):
        got = ilw.shiftmax_rows(dev(X), {"I0": I0})
        assert_same(host(got), orc.shiftmax_rows(X, I0)[0], f"edge I0={I0}")
    Xs = dev(synth.uniform_int(5, "smxs", (40, 130), -5000, 5000))
    sub = Xs[:, 3:124]  # ld 130, len 121, unaligned start
    got = ilw.shiftmax_rows(sub, {"I0": 999})
    assert_same(host(got), orc.shiftmax_rows(host(sub), 999)[0], "strided")


# ------------------------------------------------------------------------------ SD-ShiftGELU
@pytest.mark.parametrize("I0", [1, 7, 256, 1 << 10, 2047, (1 << 14) - 1])
def test_sdshiftgelu_all_int16(ilw, orc, I0):
    """Every int16 value (covers every int8 value), plus large-magnitude values."""
    x = np.arange(-(1 << 15), 1 << 15, dtype=np.int32)
    x = np.concatenate([x, np.array([1 << 23, -(1 << 23), (1 << 24) - 1, -(1 << 24) + 1, 3], np.int32)])
    got = ilw.sdshiftgelu(dev(x), {"I0": I0})
    assert_same(host(got), orc.sdshiftgelu(x, I0), f"gelu I0={I0}")


@pytest.mark.parametrize("I0", [1, 300, 1 << 10, 2047, 4000])
def test_sdshiftgelu_large_input(ilw, orc, I0):
    """Large inputs take the tabulated path (I_div(x) in shared memory for |x| <= T, constant
    beyond): every int16 value four times over, plus magnitudes far past the table's range."""
    x = np.tile(np.arange(-(1 << 15), 1 << 15, dtype=np.int32), 4)
    x = np.concatenate([x, np.array([1 << 20, -(1 << 20), (1 << 24) - 1, -(1 << 24) + 1, 40000, -40000], np.int32)])
    x = np.concatenate([x, np.zeros((-len(x)) % 4, np.int32)])
    got = ilw.sdshiftgelu(dev(x), {"I0": I0})
    assert_same(host(got), orc.sdshiftgelu(x, I0), f"gelu table I0={I0}")


def test_sdshiftgelu_unaligned_tail(ilw, orc):
    x = synth.uniform_int(6, "gt", (1003,), -4096, 4096)
    xd = dev(np.concatenate([np.zeros(1, np.int32), x]))[1:]  # 4-byte but not 16-byte aligned
    got = ilw.sdshiftgelu(xd, {"I0": 500})
    assert_same(host(got), orc.sdshiftgelu(x, 500), "gelu tail")


# ------------------------------------------------------------------------------ I-LayerNorm
@pytest.mark.parametrize("C", [1, 7, 64, 192, 384, 500, 1000, 4096])
@pytest.mark.parametrize("in_bits,out_bits,iters", [(16, 8, 10), (32, 8, 10), (32, 16, 20), (16, 16, 20)])
def test_int_layernorm(ilw, orc, C, in_bits, out_bits, iters):
    rows = 77
    lim = (1 << 14) if in_bits == 32 else 32767
    X = synth.uniform_int(7, f"ln{C}", (rows, C), -lim, lim, np.int32 if in_bits == 32 else np.int16)
    X[5] = 123  # constant row: V = 0
    X[6, :] = 0
    X[6, 0] = lim  # one dominant element
    beta, mult, shift = synth.ln_params(7, f"lnp{C}", C)
    if out_bits == 16:
        shift = shift - 7
    got = ilw.int_layernorm(dev(X), dev(beta), dev(mult), dev(shift), iters, out_bits)
    want = orc.int_layernorm(X, beta, mult, shift, iters, out_bits)
    assert_same(host(got), want, f"ln C={C}")


@pytest.mark.parametrize("rows,C,in_bits,out_bits,iters", [
    (1, 192, 16, 8, 10), (33, 384, 32, 8, 10), (1030, 256, 32, 16, 4), (70, 384, 16, 16, 3), (65, 768, 16, 8, 16), (91, 256, 16, 16, 10),
    (130, 512, 32, 8, 12)])
def test_int_layernorm_row_forms(ilw, orc, rows, C, in_bits, out_bits, iters):
    """Neighbouring rows inside and outside the range of V whose root needs no Newton steps, rows with
    V = s^2 + 2 s (the iteration alternates), rows of wide values, full and partly filled lanes."""
    rng = np.random.default_rng(rows + C)
    lim = (1 << (in_bits - 1)) - 1
    amp = np.exp(rng.uniform(0, np.log(lim if in_bits == 16 else 1 << 20), size=(rows, 1)))
    X = np.clip(np.rint(rng.standard_normal((rows, C)) * amp + rng.uniform(-1, 1, (rows, 1)) * amp), -lim, lim).astype(np.int32)
    X[::7] = 0
    X[::7, :8] = rng.integers(-1, 2, size=(len(X[::7]), 8))  # V = 0, 3, 8 = s^2 + 2 s among them
    X[3::11, 0] = -lim - 1  # the type's lowest value
    X = X.astype(np.int16 if in_bits == 16 else np.int32)
    beta, mult, shift = synth.ln_params(7, f"lnr{C}", C)
    if out_bits == 16:
        shift = shift - 7
    if rows % 2:
        shift = shift + (np.arange(C) % 3).astype(shift.dtype)  # a shift of its own for every column
    got = ilw.int_layernorm(dev(X), dev(beta), dev(mult), dev(shift), iters, out_bits)
    assert_same(host(got), orc.int_layernorm(X, beta, mult, shift, iters, out_bits), f"ln rows {rows} x {C}")


@pytest.mark.parametrize("C,in_bits", [(384, 16), (192, 32), (100, 16), (1000, 32)])
def test_int_layernorm_f16_out(ilw, orc, C, in_bits):
    """out_bits ILW_I8_IN_F16: the int8 outputs carried in float16 (the encoder's form)."""
    rows = 1000
    lim = (1 << 14) if in_bits == 32 else 32767
    X = synth.uniform_int(9, f"lnf{C}", (rows, C), -lim, lim, np.int32 if in_bits == 32 else np.int16)
    beta, mult, shift = synth.ln_params(9, f"lnpf{C}", C)
    got = ilw.int_layernorm(dev(X), dev(beta), dev(mult), dev(shift), 10, ilw.I8_IN_F16)
    assert got.dtype == torch.float16
    assert_same(host(got), orc.int_layernorm(X, beta, mult, shift, 10, 8), f"ln f16 C={C}")


# ------------------------------------------------------------------------------ attention
@pytest.mark.parametrize("B,T,H,dh,win", [(1, 17, 1, 64, 0), (2, 64, 2, 64, 0), (1, 256, 3, 64, 0),
                                          (1, 300, 2, 32, 0), (2, 100, 2, 64, 2), (1, 1600, 1, 64, 2),
                                          (1, 144, 2, 32, 3), (1, 400, 1, 64, 0)])
@pytest.mark.parametrize("form", ["int8", "f16"])
def test_attention(ilw, orc, B, T, H, dh, win, form):
    """form f16: q|k|v handed over as float16 holding the int8 values (ILW_I8_IN_F16)."""
    d = H * dh
    qkv = synth.uniform_int(8, f"qkv{T}{dh}", (B * T, 3 * d), -127, 127, np.int8)
    q_dev = dev(qkv) if form == "int8" else dev(qkv.astype(np.float16))
    for I0, sd in ((1 << 13, -1), (1 << 12, -1), (20000, 3)):
        smx = {"I0": I0, "k_inter": 16, "k_out": 8, "s_d": sd, "m_p": 4, "M_hw": 31}
        got = ilw.shiftmax_attn(q_dev, B, T, H, dh, win, smx, 3 << 29, 36)
        want = orc.attention(qkv, B, T, H, dh, win, smx, 3 << 29, 36)
        assert_same(host(got), want, f"attn T={T} win={win} I0={I0} {form}")


@pytest.mark.parametrize("B,T,H,dh,win", [(2, 1600, 2, 64, 0), (2, 1600, 2, 64, 2), (1, 300, 8, 32, 0)])
def test_attention_f16_output(ilw, orc, B, T, H, dh, win):
    """o_form ILW_I8_IN_F16 with float16 q|k|v: the encoder block's launch form."""
    d = H * dh
    qkv = synth.uniform_int(13, f"qkvo{T}{dh}", (B * T, 3 * d), -127, 127, np.int8)
    smx = {"I0": 6000, "k_inter": 16, "k_out": 8, "s_d": -1, "m_p": 4, "M_hw": 31}
    got = ilw.shiftmax_attn(dev(qkv.astype(np.float16)), B, T, H, dh, win, smx, 3 << 29, 36, o_f16=True)
    assert got.dtype == torch.float16
    assert_same(host(got), orc.attention(qkv, B, T, H, dh, win, smx, 3 << 29, 36), f"attn f16 out T={T}")


@pytest.mark.parametrize("B,T,H,dh,win", [(1, 128, 2, 64, 0), (1, 129, 1, 64, 0), (2, 257, 2, 64, 0),
                                          (1, 130, 8, 64, 0), (3, 900, 3, 64, 0), (1, 196, 1, 64, 2),
                                          (1, 1296, 1, 64, 3), (2, 6400, 1, 64, 2)])
@pytest.mark.parametrize("o_f16", [False, True])
def test_attention_tensor_memory_shapes(ilw, orc, B, T, H, dh, win, o_f16):
    """Shapes at the tensor-memory kernel's block edges with fp16-carried q|k|v: a group of exactly
    one query tile, one query past it (a tile whose warps but one have no query), several images,
    8 heads, window sides 7 (one key block of 49), 12 (two blocks of 120 keys) and 40 (14 blocks;
    the last key box reaches past the window and, for the last image, past the matrix).  Global
    groups whose last tile has at most 64 queries put two (image, head) units' last tiles in one
    CTA: T = 129, 257, 130 and 900 run that form, 3 x 3 units at T = 900 with pairs that span two
    images and a last CTA with one unit."""
    d = H * dh
    qkv = synth.uniform_int(14, f"qkvtc{T}{H}{win}", (B * T, 3 * d), -127, 127, np.int8)
    smx = {"I0": 5000, "k_inter": 16, "k_out": 8, "s_d": -1, "m_p": 4, "M_hw": 31}
    got = ilw.shiftmax_attn(dev(qkv.astype(np.float16)), B, T, H, dh, win, smx, 3 << 29, 36, o_f16=o_f16)
    want = orc.attention(qkv, B, T, H, dh, win, smx, 3 << 29, 36)
    assert_same(host(got), want, f"attn tc T={T} win={win} o_f16={o_f16}")


@pytest.mark.parametrize("I0", [1, 16, 200])
def test_attention_small_sums(ilw, orc, I0):
    """Small I0 gives row sums below 2^23, so F >= 2^(sh0) for some rows and the tensor-memory
    kernel's pass 3 takes the P form without the high-word product (every warp whose rows all allow
    it takes the other); global and windowed, fp16-carried q|k|v."""
    for B, T, H, win in ((1, 300, 2, 0), (1, 400, 1, 2)):
        d = H * 64
        qkv = synth.uniform_int(15, f"qkvsm{T}{I0}", (B * T, 3 * d), -40, 40, np.int8)
        smx = {"I0": I0, "k_inter": 16, "k_out": 8, "s_d": -1, "m_p": 4, "M_hw": 31}
        got = ilw.shiftmax_attn(dev(qkv.astype(np.float16)), B, T, H, 64, win, smx, 3 << 29, 36)
        assert_same(host(got), orc.attention(qkv, B, T, H, 64, win, smx, 3 << 29, 36), f"attn small I0={I0} T={T}")


def test_attention_extreme_scores(ilw, orc):
    """All q, k = +127 (largest scores, every row uniform) and alternating signs."""
    B, T, H, dh = 1, 130, 2, 64
    d = H * dh
    qkv = np.full((B * T, 3 * d), 127, np.int8)
    qkv[::2, d:2 * d] = -127
    smx = {"I0": 1 << 14, "k_inter": 16, "k_out": 8, "s_d": -1, "m_p": 4, "M_hw": 31}
    got = ilw.shiftmax_attn(dev(qkv), B, T, H, dh, 0, smx, 1 << 30, 33)
    assert_same(host(got), orc.attention(qkv, B, T, H, dh, 0, smx, 1 << 30, 33), "attn extreme")


def test_int_layernorm_host_time_does_not_depend_on_steps(ilw):
    """The search for the roots that need no Newton steps (long at 10 steps, short at 20) is not part of a call: 200
    calls of a short kernel take the host as long at either count (the best of 20; 14.5 and 10.2 us a call with
    the search in each)."""
    x = torch.zeros((16, 192), dtype=torch.int16, device="cuda")
    out = torch.empty((16, 192), dtype=torch.int8, device="cuda")
    ln = [dev(a) for a in synth.ln_params(7, "lnhost", 192)]

    def calls(iters):
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        for _ in range(200):
            ilw.int_layernorm(x, *ln, iters, 8, out=out)
        return time.perf_counter() - t0

    t = [(calls(10), calls(20)) for _ in range(21)][1:]  # in turn: a busy host slows both
    assert min(a for a, _ in t) < 1.2 * min(b for _, b in t)


def attention_ctas(ilw, B, T, H, dh, win, form, smx):
    """The CTAs that share a group in the resident kernel; 0: another kernel takes the problem (every problem's is the
    warp-MMA kernel under ILWDETR_ATTENTION_TC=0)."""
    ctas = ctypes.c_int32(-1)
    p = ilw.ShiftmaxT(*(smx[k] for k in ("I0", "k_inter", "k_out", "s_d", "m_p", "M_hw")))
    assert ilw.lib().ilwdetr_debug_attention_ctas(B, T, H, dh, win, 8 if form == "i8" else ilw.I8_IN_F16, ctypes.byref(p),
                                                  ctypes.byref(ctas)) == 0
    return ctas.value


def check_attention_images(ilw, orc, B, T, H, dh, win, form, smx):
    """Every image against the oracle; images beyond the first few repeat them."""
    d, n = H * dh, min(B, 3)
    qkv = synth.uniform_int(16, f"qkvr{T}{H}{dh}", (n * T, 3 * d), -90, 90, np.int8)
    full = np.concatenate([qkv.reshape(n, -1)] * (B // n + 1))[:B].reshape(B * T, 3 * d)
    got = host(ilw.shiftmax_attn(dev(full if form == "i8" else full.astype(np.float16)), B, T, H, dh, win, smx, 3 << 29, 36))
    want = orc.attention(qkv, n, T, H, dh, win, smx, 3 << 29, 36).reshape(n, -1)
    for b in range(B):
        assert_same(got.reshape(B, -1)[b], want[b % n], f"attention T={T} win={win} image {b}")


@pytest.mark.parametrize("C,lim", [(192, 1 << 20), (384, (1 << 24) - 1), (256, 1 << 23), (100, 1 << 16)])
def test_int_layernorm_wide_values(ilw, orc, C, lim):
    """int32 rows past 16 bits (up to the 2^24 that the operator takes): sums that fit 32 bits and sums that do not, of either sign, with the variance inside and
    beyond the range whose root needs no steps, and V = s^2 + 2 s."""
    rng = np.random.default_rng(C)
    X = np.concatenate([rng.integers(-lim, lim, (20, C)), lim - rng.integers(0, 3, (20, C)), rng.integers(0, 3, (20, C)) - lim,
                        np.full((20, C), -lim // 2) + rng.integers(-500, 500, (20, C))]).astype(np.int32)
    X[-1], X[-1, :3] = lim // 2, [lim // 2 + 1, lim // 2 - 1, lim // 2 + 1]  # V = 3
    beta, mult, shift = synth.ln_params(7, f"lnw{C}", C)
    for iters in (10, 20):
        got = ilw.int_layernorm(dev(X), dev(beta), dev(mult), dev(shift), iters, 8)
        assert_same(host(got), orc.int_layernorm(X, beta, mult, shift, iters, 8), f"ln wide {C} {lim} {iters}")


@pytest.mark.parametrize("B,T,H,dh,win,form,ctas", [
    (1, 1, 1, 64, 0, "f16", 1), (1, 16, 1, 64, 0, "f16", 1), (1, 33, 2, 64, 0, "f16", 1),  # one unit of 16 keys, a partial one
    (2, 257, 1, 64, 0, "f16", 4), (40, 260, 2, 32, 0, "f16", 1),  # past one MMA's 256 keys
    (30, 448, 2, 64, 0, "f16", 1), (1, 449, 1, 64, 0, "i8", 8),    # a CTA's 448 and past them
    (8, 897, 2, 64, 0, "f16", 4), (1, 1793, 1, 64, 0, "f16", 8),   # clusters of 4 and 8 CTAs
    (20, 890, 1, 64, 0, "f16", 2),                                 # of 2
    (1, 3584, 1, 64, 0, "f16", 8), (1, 3585, 1, 64, 0, "f16", 0),  # the last of a cluster of 8, and past it
    (90, 200, 2, 32, 0, "i8", 1), (82, 130, 2, 64, 0, "f16", 1),   # several jobs per CTA, units changing
    (12, 600, 2, 64, 0, "f16", 2), (5, 900, 3, 32, 0, "i8", 4),    # the same in clusters
    (2, 900, 2, 64, 2, "i8", 4), (1, 49, 2, 64, 7, "f16", 1), (2, 1764, 1, 32, 2, "f16", 4)])
def test_attention_resident_shapes(ilw, orc, B, T, H, dh, win, form, ctas):
    """The kernel whose scores stay in tensor memory, at the edges of its tiles and of its split over a cluster."""
    smx = {"I0": 4000, "k_inter": 16, "k_out": 8, "s_d": -1, "m_p": 4, "M_hw": 31}
    assert attention_ctas(ilw, B, T, H, dh, win, form, smx) == (ctas if TENSOR_MEMORY else 0)
    check_attention_images(ilw, orc, B, T, H, dh, win, form, smx)


@pytest.mark.parametrize("B,T,H,dh,win,form,resident", [
    (600, 64, 2, 64, 0, "f16", False), (600, 64, 2, 64, 0, "i8", False), (200, 16, 2, 32, 0, "f16", False),
    (100, 63, 2, 64, 0, "f16", False), (200, 1, 2, 64, 0, "i8", False), (4, 1600, 3, 64, 10, "f16", False),  # one key tile
    (1, 64, 3, 32, 0, "i8", False), (1, 128, 3, 32, 0, "i8", False), (300, 65, 2, 64, 0, "f16", True),
    (100, 100, 6, 64, 0, "f16", True), (100, 192, 6, 32, 0, "f16", False), (8, 300, 8, 32, 0, "i8", True),
    (16, 2300, 6, 64, 0, "f16", False), (16, 1600, 6, 64, 0, "f16", True),
    (1, 33, 2, 32, 0, "f16", False), (1, 448, 1, 64, 0, "f16", True), (1, 897, 1, 64, 0, "f16", True),
    (90, 40, 2, 32, 0, "i8", False), (41, 130, 2, 64, 0, "f16", True), (1, 5329, 1, 64, 1, "f16", False),
    (1, 441, 2, 64, 21, "f16", False)])
def test_attention_choice(ilw, orc, B, T, H, dh, win, form, resident):
    """The kernel that was faster where all were timed, and the result of the short groups, whose kernel depends on the number
    of groups and on the form of q|k|v."""
    smx = {"I0": 4000, "k_inter": 16, "k_out": 8, "s_d": -1, "m_p": 4, "M_hw": 31}
    assert (attention_ctas(ilw, B, T, H, dh, win, form, smx) > 0) == (resident and TENSOR_MEMORY)
    if B * T < 10000 or T <= 300 or win:
        check_attention_images(ilw, orc, B, T, H, dh, win, form, smx)


@pytest.mark.parametrize("I0,k_inter,k_out,m_p", [(1, 16, 8, 4), (3, 10, 4, 0), (700, 0, 8, 4), (16384, 16, 8, 4),
                                                  (32767, 15, 7, 4), (32767, 16, 8, 16), (9000, 16, 1, 31)])
def test_attention_resident_parameters(ilw, orc, I0, k_inter, k_out, m_p):
    """Its Shiftmax parameters over their range: sums of four and of two values in 32 bits, every form
    of the output (one and two outputs per word, the 64-bit product), and shifts of the output
    requantisation on both sides of 33; int8 outputs with rows that no vector store fits."""
    B, T, H = 1, 210, 1
    qkv = synth.uniform_int(17, f"qkvp{I0}{k_inter}", (B * T, 192), -60, 60, np.int8)
    smx = {"I0": I0, "k_inter": k_inter, "k_out": k_out, "s_d": -1, "m_p": m_p, "M_hw": 31}
    out = torch.zeros((B * T, 70), dtype=torch.int8, device="cuda")
    for s_o in (30, 36):
        ilw.shiftmax_attn(dev(qkv.astype(np.float16)), B, T, H, 64, 0, smx, 3 << 28, s_o, out=out[:, 3:67])
        want = orc.attention(qkv, B, T, H, 64, 0, smx, 3 << 28, s_o)
        assert_same(host(out[:, 3:67]), want, f"resident I0={I0} k={k_inter} s_o={s_o}")
        assert not bool(out[:, :3].any()) and not bool(out[:, 67:].any())


# ------------------------------------------------------------------------------ split conv
def test_split_conv(ilw, orc):
    M, N, Ks = 333, 256, (384, 384, 384, 384)
    Xs = [synth.uniform_int(9, f"sx{i}", (M, k), -127, 127, np.int8) for i, k in enumerate(Ks)]
    Ws = [synth.uniform_int(9, f"sw{i}", (N, k), -127, 127, np.int8) for i, k in enumerate(Ks)]
    bias = synth.uniform_int(9, "sb", (N,), -(1 << 15), 1 << 15)
    mult = synth.uniform_int(9, "sm", (N,), 1 << 30, (1 << 31) - 1)
    shift = np.full(N, 40, np.int32)
    m_b = [1 << 30, 3 << 28, 1 << 29, 1 << 30]
    s_b = [30, 31, 31, 32]
    got = ilw.split_conv([dev(x) for x in Xs], [ilw.pack_weight(dev(w)) for w in Ws], N, m_b, s_b,
                         dev(bias), dev(mult), dev(shift))
    want = orc.split_conv(Xs, Ws, m_b, s_b, bias, mult, shift)
    assert_same(host(got), want, "split conv")


@pytest.mark.parametrize("M,N,Ks,s_b", [(100, 64, (64,), [27]), (130, 200, (384, 80, 1024), [26, 33, 45]),
                                        (9900, 136, (64, 128), [30, 28])])
def test_split_conv_forms(ilw, orc, M, N, Ks, s_b):
    """Tiles of 64 and 128 columns, ragged sizes, branch shifts from 26 on."""
    Xs = [synth.uniform_int(19, f"sx{i}{M}", (M, k), -127, 127, np.int8) for i, k in enumerate(Ks)]
    Ws = [synth.uniform_int(19, f"sw{i}{N}", (N, k), -127, 127, np.int8) for i, k in enumerate(Ks)]
    Xs[0][0], Ws[0][0], Ws[0][1] = 127, 127, -127  # the largest accumulators
    bias = synth.uniform_int(19, f"sb{N}", (N,), -(1 << 15), 1 << 15)
    mult = synth.uniform_int(19, f"sm{N}", (N,), 1 << 30, (1 << 31) - 1)
    shift = np.full(N, 45, np.int32)
    m_b = [(1 << 24) + 12345 * i if s < 29 else 3 << 28 for i, s in enumerate(s_b)]
    got = ilw.split_conv([dev(x) for x in Xs], [ilw.pack_weight(dev(w)) for w in Ws], N, m_b, s_b, dev(bias), dev(mult), dev(shift))
    assert_same(host(got), orc.split_conv(Xs, Ws, m_b, s_b, bias, mult, shift), "split conv")


# ------------------------------------------------------------------------------ deformable sampling
def test_deform_attn(ilw, orc):
    B, Q, H, L, P, dh = 2, 300, 8, 3, 4, 32
    hw = [(80, 80), (40, 40), (20, 20)]
    S = sum(h * w for h, w in hw)
    value = synth.uniform_int(10, "dv", (B, S, H * dh), -127, 127, np.int8)
    ref = synth.uniform_int(10, "dr", (B, Q, 2), 0, 65535)
    off = synth.uniform_int(10, "do", (B, Q, H, L, P, 2), -(8 << 8), 8 << 8)
    off[0, 0] = -(1 << 20)  # every sample of one query far outside
    w = synth.uniform_int(10, "dw", (B, Q, H, L * P), 0, 40, np.uint8)
    got = ilw.deform_attn(dev(value), hw, dev(ref), dev(off), dev(w), 3 << 29, 36)
    want = orc.deform_attn(value, hw, ref, off, w, 3 << 29, 36)
    assert_same(host(got), want, "deform")


# ------------------------------------------------------------------------------ block
@pytest.mark.parametrize("cfg", ["block256_literal", "block256_calibrated", "small_window"])
def test_block_forward(ilw, orc, cfg):
    if cfg.startswith("block256"):
        B, T, d, H, F, win, mode = 1, 256, 192, 3, 768, 0, cfg.split("_")[1]
    else:
        B, T, d, H, F, win, mode = 2, 400, 128, 2, 256, 2, "calibrated"
    bp = synth.block_params(0, 0, d, H, F, win, mode)
    x = synth.block_input(0, B, T, d)
    bw = ilw.BlockWeights(bp)
    ws = torch.empty(ilw.block_workspace_bytes(B, T, d, F), dtype=torch.uint8, device="cuda")
    y = ilw.block_forward(bw, dev(x), B, T, ws)
    y_ref, taps = orc.block_forward(bp, x, B, T, taps=True)
    assert_same(host(y), y_ref, f"block {cfg}")
    # every intermediate, through the op-level entry points
    t = bw.t
    a1 = ilw.int_layernorm(dev(x), t["ln1_beta"], t["ln1_mult"], t["ln1_shift"], 10, 8)
    assert_same(host(a1), taps["a1"], "a1")
    qkv = ilw.gemm_requant(a1, t["w_qkv_p"], 3 * d, t["b_qkv"], t["m_qkv"], t["s_qkv"], 8)
    assert_same(host(qkv), taps["qkv"], "qkv")
    o = ilw.shiftmax_attn(qkv, B, T, H, d // H, win, bp["smx"], bp["m_o"], bp["s_o"])
    assert_same(host(o), taps["o"], "attention")
    x1 = ilw.gemm_requant(o, t["w_proj_p"], d, t["b_proj"], t["m_proj"], t["s_proj"], 16, res=dev(x),
                          m_r=bp["m_r1"], s_r=bp["s_r1"])
    assert_same(host(x1), taps["x1"], "x1")
    a2 = ilw.int_layernorm(x1, t["ln2_beta"], t["ln2_mult"], t["ln2_shift"], 10, 8)
    assert_same(host(a2), taps["a2"], "a2")
    h = ilw.gemm_gelu(a2, t["w_fc1_p"], F, t["b_fc1"], t["m_fc1"], t["s_fc1"],
                      {"I0": bp["gelu_I0"]}, bp["m_g"], bp["s_g"])
    assert_same(host(h), taps["h"], "h")
    y2 = ilw.gemm_requant(h, t["w_fc2_p"], d, t["b_fc2"], t["m_fc2"], t["s_fc2"], 16, res=x1,
                          m_r=bp["m_r2"], s_r=bp["s_r2"])
    assert_same(host(y2), y_ref, "y via ops")
    ilw.device_status()


@pytest.mark.parametrize("M,N,K,out_bits,res_rows,mult", [
    (130, 384, 384, 16, 130, 0), (300, 384, 1536, 16, 300, 0), (97, 104, 128, 16, 32, 0), (200, 136, 256, 16, 50, 0),
    (33, 576, 384, 8, 0, 0), (257, 200, 1104, 8, 0, 0), (129, 1152, 384, 108, 0, 0), (64, 130, 64, 108, 0, 0),
    (2500, 576, 384, 108, 0, 0), (2500, 584, 320, 8, 0, 0), (3300, 384, 1536, 16, 3300, 0),
    (140, 256, 256, 8, 0, 1 << 30), (140, 384, 320, 108, 0, 3 << 28), (70, 48, 192, 8, 70, 0)])
@pytest.mark.parametrize("a_f16,spread", [(False, False), (True, False), (True, True), (False, True)])
def test_gemm_epilogue_forms(ilw, orc, M, N, K, out_bits, res_rows, mult, a_f16, spread):
    """One shift for all columns, or (spread) one each from 29 on: int8 results in floats with the integers for
    values near a half (mult: a coarse scale, whose results are often exact halves), accumulators inside and
    beyond 2^22, residuals of whole and broadcast tables (32-row boxes that wrap or not), in place, and columns
    past the last tile."""
    A = synth.uniform_int(21, f"ef{M}{K}", (M, K), -127, 127, np.int8)
    W, b, m, s = synth.gemm_params(21, f"efW{N}{K}", N, K, 60.0 if out_bits != 16 else 9000.0, 30.0, "literal")
    A[M // 2], W[N // 3] = 127, 127  # accumulators up to 127^2 K
    s = (29 + np.arange(N) % 14).astype(s.dtype) if spread else np.full_like(s, s[0])
    if mult:
        m = np.full_like(m, mult)
        m[::5] = -m[::5]
        s = np.full_like(s, 42) if not spread else s
    A_d = dev(A.astype(np.float16) if a_f16 else A)
    args = (A_d, ilw.pack_weight(dev(W)), N, dev(b), dev(m), dev(s), out_bits)
    if res_rows:
        res = synth.uniform_int(21, f"efr{res_rows}{N}", (res_rows, N), -32767, 32767, np.int16)
        want = orc.gemm_requant(A, W, b, m, s, out_bits, res, 3 << 28, 30)
        r_d = dev(res)
        assert_same(host(ilw.gemm(*args, res=r_d, m_r=3 << 28, s_r=30)), want, "residual")
        if res_rows == M and out_bits == 16:  # in place
            ilw.gemm(*args, res=r_d, m_r=3 << 28, s_r=30, out=r_d)
            assert_same(host(r_d), want, "residual in place")
    else:
        want = orc.gemm_requant(A, W, b, m, s, 8, None, 0, 0)
        assert_same(host(ilw.gemm(*args)), want, "int8")


@pytest.mark.parametrize("M,N,K,a_f16,out_bits", [
    (30000, 1152, 64, False, 8), (30000, 1536, 192, False, 8),  # three groups of 32 columns a warp
    (14400, 576, 192, True, 108), (40000, 640, 192, True, 108), (40000, 640, 320, True, 8),  # one, resident weights
    (40000, 256, 1104, True, 8)])                               # one, streamed weights
def test_gemm_store_boxes_over_tiles(ilw, orc, M, N, K, a_f16, out_bits):
    """Results stored through shared memory, an odd number of column groups in a warp's part of a tile and four or
    more tiles a CTA, so that a store box is filled again while earlier stores may be under way: every element of
    repeated calls (1000 distinct rows, repeated)."""
    n = 1000
    A = synth.uniform_int(23, f"sb{K}", (n, K), -127, 127, np.int8)
    W, b, m, s = synth.gemm_params(23, f"sbW{N}{K}", N, K, 60.0, 30.0, "literal")
    want = dev(orc.gemm_requant(A, W, b, m, s, 8, None, 0, 0).astype(np.float16 if out_bits == 108 else np.int8))
    A_d = dev(A.astype(np.float16) if a_f16 else A).repeat(M // n + 1, 1)[:M].contiguous()
    Wp, b, m, s = ilw.pack_weight(dev(W)), dev(b), dev(m), dev(s)
    for _ in range(5):
        got = ilw.gemm(A_d, Wp, N, b, m, s, out_bits)
        for r in range(0, M, n):
            assert torch.equal(got[r:r + n], want[:min(n, M - r)]), r
    ilw.device_status()


@pytest.mark.parametrize("M,N,K,out_bits,res", [
    (5000, 200, 768, 16, ""), (5000, 200, 768, 8, "r"), (5000, 200, 768, 16, "r"), (5000, 200, 768, 16, "odd"), (4900, 136, 1104, 16, ""),
    (9700, 136, 2112, 16, "r"), (9700, 136, 2112, 8, ""), (5000, 200, 768, 32, ""), (5000, 200, 128, 32, ""), (9700, 72, 2112, 32, "")])
@pytest.mark.parametrize("spread", [False, True])
def test_gemm_column_parts(ilw, orc, M, N, K, out_bits, res, spread):
    """128-wide tiles of fp16 rows with two column parts (raw accumulators; streamed weights without a residual box,
    with int8 residuals, with three accumulators) and with four (residual by TMA), one shift or (spread) one for every
    column, columns past the last tile, residual rows that TMA takes and (odd) does not."""
    n = 400
    A = synth.uniform_int(25, f"cp{K}", (n, K), -127, 127, np.int8)
    W, b, m, s = synth.gemm_params(25, f"cpW{N}{K}", N, K, 60.0, 30.0 if out_bits == 8 else 9000.0, "literal")
    A[n // 2], W[N // 3] = 127, 127  # accumulators up to 127^2 K
    s = (29 + np.arange(N) % 14).astype(s.dtype) if spread else np.full_like(s, s[0])
    R = synth.uniform_int(25, f"cpr{N}", (n, N), -32768, 32767, np.int16) if res else None
    want = dev(orc.gemm_requant(A, W, b, m, s, out_bits, R, 3 << 28, 30))
    kw = {}
    if res:
        r_d = torch.zeros((M, N + 3 if res == "odd" else N), dtype=torch.int16, device="cuda")[:, :N]
        r_d[:] = dev(R).repeat(M // n + 1, 1)[:M]
        kw = dict(res=r_d, m_r=3 << 28, s_r=30)
    A_d = dev(A.astype(np.float16)).repeat(M // n + 1, 1)[:M].contiguous()
    got = ilw.gemm(A_d, ilw.pack_weight(dev(W)), N, dev(b), None if out_bits == 32 else dev(m), None if out_bits == 32 else dev(s),
                   out_bits, **kw)
    for r in range(0, M, n):
        assert torch.equal(got[r:r + n].to(torch.int32), want[:min(n, M - r)].to(torch.int32)), r


@pytest.mark.parametrize("s_r", [1, 16, 17, 46, 47, 48, 62])
@pytest.mark.parametrize("M,N,a_f16", [(70, 200, False), (4000, 384, True)])  # 64-wide tiles, resident weights
def test_gemm_residual_shifts(ilw, orc, M, N, a_f16, s_r):
    """The residual's shift on both sides of the 32-bit form's range and at its ends, with the largest residuals and
    multipliers of either sign; accumulators whose own term nears 2^31 where the shifts are small."""
    A = synth.uniform_int(24, f"rs{M}", (M, 64), -127, 127, np.int8)
    W, b, m, s = synth.gemm_params(24, f"rsW{N}", N, 64, 60.0, 9000.0, "literal")
    res = synth.uniform_int(24, f"rsr{M}{N}", (M, N), -32768, 32767, np.int16)
    res[:, :3] = [-32768, 32767, -1]
    A_d, Wp, r_d = dev(A.astype(np.float16) if a_f16 else A), ilw.pack_weight(dev(W)), dev(res)
    for out_bits in (8, 16):
        for m_r, shift in ((1 << 30, s), (-(1 << 31), s), ((1 << 31) - 1, np.where(np.arange(N) % 2, 18, s).astype(s.dtype))):
            want = orc.gemm_requant(A, W, b, m, shift, out_bits, res, m_r, s_r)
            got = ilw.gemm(A_d, Wp, N, dev(b), dev(m), dev(shift), out_bits, res=r_d, m_r=m_r, s_r=s_r)
            assert_same(host(got), want, f"out {out_bits} m_r={m_r} s_r={s_r}")


@pytest.mark.parametrize("M,N,K", [(2500, 576, 384), (2500, 1024, 256), (700, 1024, 256), (129, 200, 64)])
@pytest.mark.parametrize("a_f16,out_bits", [(True, 108), (True, 8), (False, 8)])
def test_gemm_gelu_widths(ilw, orc, M, N, K, a_f16, out_bits):
    """SD-ShiftGELU through tiles of 192, 128 and 64 columns."""
    A = synth.uniform_int(22, f"gw{M}{K}", (M, K), -127, 127, np.int8)
    W, b, m, s = synth.gemm_params(22, f"gwW{N}{K}", N, K, 60.0, 900.0, "calibrated")
    gelu = {"I0": 500, "k_inter": 16, "k_out": 8}
    got = ilw.gemm(dev(A.astype(np.float16) if a_f16 else A), ilw.pack_weight(dev(W)), N, dev(b), dev(m), dev(s), out_bits,
                   gelu=gelu, m_g=5 << 28, s_g=41)
    h = orc.sdshiftgelu(orc.gemm_requant(A, W, b, m, s, 16), gelu["I0"]).astype(np.int64)
    want = np.clip((h * (5 << 28) + (1 << 40)) >> 41, -127, 127)
    assert_same(host(got), want, "gelu")
    assert len(np.unique(want)) > 20


# ------------------------------------------------------------- launches that overlap the one before
@pytest.mark.parametrize("M", [40, 3000])
def test_launches_follow_one_another(ilw, M):
    """A kernel may start before the one ahead of it on the stream has written its results: chains in which
    every launch reads what the last one wrote, buffers are rewritten in place and reused, and copies and
    a forked stream come between, back to back, and recorded as a graph and replayed, against the same
    chain with a synchronisation after every call."""
    N = 192
    x0 = dev(synth.uniform_int(11, f"chain{M}", (M, N), -3000, 3000, np.int16))
    W, b, m, s = synth.gemm_params(11, "chainW", N, N, 73.0, 3000.0, "literal")
    Wp, b, m, s = ilw.pack_weight(dev(W)), dev(b), dev(m), dev(s)
    ln = [dev(a) for a in synth.ln_params(11, "chainln", N)]
    x, x8, r8, y, c = (torch.empty((M, N), dtype=t, device="cuda")
                       for t in (torch.int16, torch.int8, torch.int8, torch.int16, torch.int16))
    side = torch.cuda.Stream()

    def chain(sync=lambda: None):
        x.copy_(x0), sync()
        for i in range(6):
            ilw.int_layernorm(x, *ln, out=x8), sync()
            main = torch.cuda.current_stream()
            side.wait_stream(main)
            with torch.cuda.stream(side):  # the fork reads x8 while the main stream does
                ilw.relu_i8(x8, out=r8), sync()
            ilw.gemm_requant(x8, Wp, N, b, m, s, 16, res=x, m_r=3 << 28, s_r=30, out=x), sync()
            main.wait_stream(side)
            ilw.gemm_requant(r8, Wp, N, b, m, s, 16, out=y), sync()
            c.copy_(y), sync()
            ilw.requant(x, 1 << 30, 31, Z=c, m2=1 << 30, s2=31, out_bits=16, out=x), sync()
        return x.clone()

    want = chain(torch.cuda.synchronize)
    assert len(torch.unique(want)) > 100
    for _ in range(20):
        got = chain()
        torch.cuda.synchronize()
        assert torch.equal(got, want)
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        got = chain()
    for _ in range(20):
        g.replay()
        torch.cuda.synchronize()
        assert torch.equal(got, want)
