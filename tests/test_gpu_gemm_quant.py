"""GPU parity of the product with the fused quantizing epilogue (mxfp4_gemm_quant).

The bf16 tile the kernel emits is held against the FP64 oracle product within the product's bound; the codes and
scales it emits are held, bit for bit, against the oracle's quantizers applied to THAT bf16 tile (the quantization
comes after the cast, so it cannot be pinned to the FP64 product itself)."""
import math

import numpy as np
import pytest
import torch

import oracle as orc
import workloads
from util import assert_qmat_equal, check_gemm_bound, numpy_to_qmat, qmat_to_numpy, to_dev_bf16

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mx():
    import paper_2502_20853_b200 as m
    m.lib()
    assert torch.cuda.is_available()
    return m


def rand_operand(rng, rows, kc, lo=123, hi=131):
    c = rng.integers(0, 16, size=(rows, kc)).astype(np.uint8)
    p = (c[:, 0::2] | (c[:, 1::2] << 4)).astype(np.uint8)
    s = rng.integers(lo, hi, size=(rows, kc // 32)).astype(np.uint8)
    return p, s


def operands(mx, M, N, K, seed):
    rng = np.random.default_rng(seed)
    pa, sa = rand_operand(rng, M, K)
    pb, sb = rand_operand(rng, N, K)
    return (pa, sa, pb, sb), numpy_to_qmat(mx, pa, sa), numpy_to_qmat(mx, pb, sb)


def bf16_tensor(M, N, pad=0):
    """[M, N] bf16 view of a wider buffer filled with a sentinel, to see writes beyond N."""
    big = torch.full((M, N + pad), 7.0, dtype=torch.bfloat16, device="cuda")
    return big, big[:, :N]


# one tile, several tiles, ragged in M and N (multiples of 32 only), short and long contractions
SHAPES = [(128, 128, 64), (256, 256, 512), (384, 320, 192), (160, 96, 64), (1024, 768, 1536), (512, 1152, 384)]


@pytest.mark.parametrize("M,N,K", SHAPES)
@pytest.mark.parametrize("mode", ["2axis_sr", "chain", "rne_rne", "row_only", "t_only"])
def test_quantizing_epilogue_identity(mx, M, N, K, mode):
    ops, a, b = operands(mx, M, N, K, M + 3 * N + K)
    st = mx.new_status()
    big, z = bf16_tensor(M, N, 64)
    seed = 0xABC0 + M
    qp_row = {"2axis_sr": (0, 1, seed, 3), "chain": (0, 0, 0, 0), "rne_rne": (0, 0, 0, 0), "row_only": (0, 1, seed, 3), "t_only": None}[mode]
    qp_t = {"2axis_sr": (0, 1, seed, 5), "chain": (0, 1, seed, 6), "rne_rne": (1, 0, 0, 0), "row_only": None, "t_only": (0, 1, seed, 5)}[mode]
    epi = mx.Epilogue(z=z, zq=mx.QMat(M, N) if qp_row else None, qp_row=qp_row or (0, 0, 0, 0),
                      zq_t=mx.QMat(N, M) if qp_t else None, qp_t=qp_t or (0, 0, 0, 0), chain=(mode == "chain"))
    mx.gemm_quant(a, b, epi, dev_status=st)
    torch.cuda.synchronize()
    assert int(st.item()) == 0
    assert (big[:, N:] == 7.0).all()
    zf = z.float().cpu().numpy()
    dref, tref = orc.gemm(*ops)
    check_gemm_bound(zf, dref, tref, True, "Z")
    if qp_row:
        pr, sr, _ = orc.quantize(zf, scale_mode=qp_row[0], rounding=qp_row[1], seed=qp_row[2], stream_id=qp_row[3])
        assert_qmat_equal(epi.zq, pr, sr, "row-wise codes of Z")
    if qp_t:
        src = orc.dequantize(pr, sr) if mode == "chain" else zf
        pt, s_t, _ = orc.quantize(src, transpose=True, scale_mode=qp_t[0], rounding=qp_t[1], seed=qp_t[2], stream_id=qp_t[3])
        assert_qmat_equal(epi.zq_t, pt, s_t, "transposed codes of Z")


def test_quantizing_epilogue_gelu_with_bias_keeps_y(mx):
    M, N, K = 384, 640, 256
    ops, a, b = operands(mx, M, N, K, 5)
    rng = np.random.default_rng(6)
    bias = workloads.round_to_bf16((rng.standard_normal(N) * 2).astype(np.float32))
    y = torch.empty((M, N), dtype=torch.bfloat16, device="cuda")
    z = torch.empty((M, N), dtype=torch.bfloat16, device="cuda")
    seed = 99
    epi = mx.Epilogue(hook=mx.HOOK_GELU, y=y, z=z, zq=mx.QMat(M, N), qp_row=(0, 0, 0, 0), zq_t=mx.QMat(N, M), qp_t=(0, 1, seed, 6), chain=True)
    st = mx.new_status()
    mx.gemm_quant(a, b, epi, bias=to_dev_bf16(bias.reshape(1, -1)).reshape(-1), dev_status=st)
    torch.cuda.synchronize()
    assert int(st.item()) == 0
    dref, tref = orc.gemm(*ops)
    yf = y.float().cpu().numpy().astype(np.float64)
    want = dref + bias
    tol = tref * 2.0 ** -20 + np.abs(want) * 2.0 ** -23
    lo = np.minimum(workloads.round_to_bf16((want - tol).astype(np.float32)), want - tol)
    hi = np.maximum(workloads.round_to_bf16((want + tol).astype(np.float32)), want + tol)
    assert ((yf >= lo) & (yf <= hi)).all(), "Y = bf16(product + bias)"
    # Z = bf16(GELU(Y)): the FP32 evaluation (absolute error below 1e-6 |y|) may land on the neighbouring bf16 value
    erf = np.vectorize(math.erf)
    g = 0.5 * yf * (1.0 + erf(yf / math.sqrt(2.0)))
    zf = z.float().cpu().numpy().astype(np.float64)
    assert (np.abs(zf - g) <= np.abs(g) * 2.0 ** -8 + np.abs(yf) * 2.0 ** -20).all(), "Z = bf16(GELU(Y))"
    pr, sr, _ = orc.quantize(zf.astype(np.float32))
    assert_qmat_equal(epi.zq, pr, sr, "Q1 of the next layer")
    pt, s_t, _ = orc.quantize(orc.dequantize(pr, sr), transpose=True, rounding=1, seed=seed, stream_id=6)
    assert_qmat_equal(epi.zq_t, pt, s_t, "Q6 of the next layer")


# one kernel or two, by 128 x 128 tiles on 148 SMs.  Y and Z stored: two from four per SM on (627; 592 with ragged last tiles; 588: one).  Y
# alone: two from twelve per SM on (1776, also ragged; 1764: one; 592: one), and from four on where the contraction is longer than 1024
@pytest.mark.parametrize("M,N,K,with_z,launches", [
    (4128, 2336, 64, True, 2), (18912, 480, 64, True, 2), (18784, 480, 64, True, 1), (18944, 512, 64, False, 1), (18912, 512, 64, False, 1),
    (18944, 1536, 64, False, 2), (18912, 1504, 64, False, 2), (18784, 1504, 64, False, 1), (18912, 480, 1056, False, 2)])
def test_gelu_chain_of_many_tiles(mx, M, N, K, with_z, launches):
    """The product and the quantization behind GELU in one kernel or in two, which reads Y back: sizes on both sides of the lines
    and partial tiles, Y with a leading dimension of its own."""
    ops, a, b = operands(mx, M, N, K, 11)
    big = torch.full((M, N + 16), 7.0, dtype=torch.bfloat16, device="cuda")
    y = big[:, :N]
    z = torch.empty((M, N), dtype=torch.bfloat16, device="cuda") if with_z else None
    epi = mx.Epilogue(hook=mx.HOOK_GELU, y=y, z=z, zq=mx.QMat(M, N), zq_t=mx.QMat(N, M), qp_t=(0, 1, 5, 6), chain=True)
    st = mx.new_status()
    n0 = mx.launch_count()
    mx.gemm_quant(a, b, epi, dev_status=st)
    assert mx.launch_count() == n0 + launches
    torch.cuda.synchronize()
    assert int(st.item()) == 0 and bool((big[:, N:] == 7.0).all())
    assert torch.equal(y, mx.gemm(a, b))
    yd = y.double()
    g = 0.5 * yd * (1.0 + torch.erf(yd / math.sqrt(2.0)))
    if with_z:
        assert bool(((z.double() - g).abs() <= g.abs() * 2.0 ** -8 + yd.abs() * 2.0 ** -20).all())
    else:   # the codes of Z stand for it: dequantized, they are within half a step of the group's grid (6 * 2^s >= the maximum)
        gm = g.abs().reshape(M, N // 32, 32).amax(2, keepdim=True)
        d = (mx.dequantize(epi.zq).double() - g).abs().reshape(M, N // 32, 32)
        assert bool((d <= gm * (1.01 / 3)).all())
        z = None
    if z is not None:
        q, qt = mx.quantize_chain(z, seed=5)
        for got, want in ((epi.zq, q), (epi.zq_t, qt)):
            assert torch.equal(got.data, want.data) and torch.equal(got.scales_linear(), want.scales_linear())
    else:
        qt = mx.quantize_t(epi.zq, rounding=1, seed=5, stream_id=6)
        assert torch.equal(epi.zq_t.data, qt.data) and torch.equal(epi.zq_t.scales_linear(), qt.scales_linear())


def test_quantizing_epilogue_multiply_is_exact(mx):
    """dX times the derivative of the activation, then Q3 / Q5 of the previous layer: the product of two bf16 values is
    exact in FP32, so Z = bf16(Y * aux) is reproducible bit for bit from the Y the kernel emitted."""
    M, N, K = 512, 384, 1536
    ops, a, b = operands(mx, M, N, K, 7)
    rng = np.random.default_rng(8)
    aux = workloads.round_to_bf16(rng.uniform(-0.2, 1.1, size=(M, N)).astype(np.float32))
    auxd = to_dev_bf16(aux)
    y = torch.empty((M, N), dtype=torch.bfloat16, device="cuda")
    z = torch.empty((M, N), dtype=torch.bfloat16, device="cuda")
    seed = 1234
    epi = mx.Epilogue(hook=mx.HOOK_MULTIPLY, aux=auxd, y=y, z=z, zq=mx.QMat(M, N), qp_row=(0, 1, seed, 3), zq_t=mx.QMat(N, M), qp_t=(0, 1, seed, 5))
    st = mx.new_status()
    mx.gemm_quant(a, b, epi, dev_status=st)
    torch.cuda.synchronize()
    assert int(st.item()) == 0
    dref, tref = orc.gemm(*ops)
    yf = y.float().cpu().numpy()
    check_gemm_bound(yf, dref, tref, True, "Y")
    zref = workloads.round_to_bf16(yf * aux)          # float32 product of bf16 values: exact, then one rounding
    zf = z.float().cpu().numpy()
    assert (zf.view(np.uint32) == zref.view(np.uint32)).all(), "Z = bf16(Y * aux)"
    assert_qmat_equal(epi.zq, *orc.quantize(zf, rounding=1, seed=seed, stream_id=3)[:2], "Q3")
    assert_qmat_equal(epi.zq_t, *orc.quantize(zf, transpose=True, rounding=1, seed=seed, stream_id=5)[:2], "Q5")


def test_quantizing_epilogue_equals_the_standalone_quantizers(mx):
    """At a size the oracle would take long on: the fused results against mxfp4_quantize_chain / _2axis on the same Z."""
    M, N, K = 4096, 1536, 384
    g = torch.Generator(device="cuda").manual_seed(3)
    a, b = mx.QMat(M, K), mx.QMat(N, K)
    for q in (a, b):
        q.data.copy_(torch.randint(0, 256, q.data.shape, dtype=torch.uint8, device="cuda", generator=g))
        q.scales.copy_(torch.randint(124, 130, q.scales.shape, dtype=torch.uint8, device="cuda", generator=g))
    seed = 4242
    for chain, qp_row, qp_t in ((True, (0, 0, 0, 0), (0, 1, seed, 6)), (False, (0, 1, seed, 3), (0, 1, seed, 5))):
        z = torch.empty((M, N), dtype=torch.bfloat16, device="cuda")
        epi = mx.Epilogue(z=z, zq=mx.QMat(M, N), qp_row=qp_row, zq_t=mx.QMat(N, M), qp_t=qp_t, chain=chain)
        mx.gemm_quant(a, b, epi)
        assert torch.equal(z, mx.gemm(a, b)), "the bf16 tile equals the plain product's"
        if chain:
            q, qt = mx.quantize_chain(z, seed=seed)
        else:
            q, qt = mx.quantize_2axis(z, qp_row, qp_t)
        assert torch.equal(epi.zq.data, q.data) and torch.equal(epi.zq.scales, q.scales)
        assert torch.equal(epi.zq_t.data, qt.data) and torch.equal(epi.zq_t.scales, qt.scales)


@pytest.mark.parametrize("M,N", [(384, 256), (6400, 384)])   # one group of epilogue warps, two (150 tiles)
def test_multiply_by_any_bf16_value(mx, M, N):
    """Z = bf16(Y * aux), exact before its one rounding, over all bf16 values of aux (subnormal ones, infinities, NaN) and Y over
    many binades: products that are subnormal, tie at the smallest ones, vanish, overflow, or are no number."""
    rng = np.random.default_rng(N)
    c = rng.integers(0, 16, size=(M, 32)).astype(np.uint8)
    unit = np.zeros((N, 32), np.uint8)
    unit[np.arange(N), np.arange(N) % 32] = 2                       # 1.0: Y[m, n] = A[m, n % 32]
    pack = lambda v: (v[:, 0::2] | (v[:, 1::2] << 4)).astype(np.uint8)  # noqa: E731
    a = numpy_to_qmat(mx, pack(c), rng.integers(8, 247, size=(M, 1)).astype(np.uint8))
    b = numpy_to_qmat(mx, pack(unit), np.full((N, 1), 127, np.uint8))
    bits = rng.integers(0, 1 << 16, size=(M, N)).astype(np.int32)
    bits[:, ::7] = rng.choice([0, 0x8000, 1, 0x8001, 0x7F, 0x80, 0x7F7F, 0xFF7F, 0x7F80, 0xFF80, 0x7FC0, 0xFF81], size=bits[:, ::7].shape)
    aux = torch.from_numpy(bits.astype(np.uint16).view(np.int16)).view(torch.bfloat16).cuda()
    y = mx.gemm(a, b)
    z = torch.empty((M, N), dtype=torch.bfloat16, device="cuda")
    epi = mx.Epilogue(hook=mx.HOOK_MULTIPLY, aux=aux, z=z, zq=mx.QMat(M, N), qp_row=(0, 1, 9, 3), zq_t=mx.QMat(N, M), qp_t=(0, 1, 9, 5))
    st = mx.new_status()
    mx.gemm_quant(a, b, epi, dev_status=st)
    torch.cuda.synchronize()
    assert int(st.item()) == mx.DEV_NONFINITE
    with np.errstate(invalid="ignore", over="ignore"):
        p = y.double().cpu().numpy() * aux.double().cpu().numpy()   # 16 bits: exact
        ulp = np.ldexp(1.0, np.maximum(np.frexp(p)[1] - 1, -126) - 7)
        want = np.where(np.isfinite(p), np.rint(p / ulp) * ulp, p)
        want[np.abs(want) >= 2.0 ** 128] *= np.inf
    zf = z.double().cpu().numpy()
    assert (((np.abs(want) < 2.0 ** -126) & (want != 0)).sum() > 100 and (want == 0).sum() > 100 and (np.isinf(want) & np.isfinite(p)).sum() > 100 and
            np.isnan(want).sum() > 100)
    assert np.array_equal(zf, want, equal_nan=True)
    q, qt = mx.quantize_2axis(z, (0, 1, 9, 3), (0, 1, 9, 5))
    for got, ref in ((epi.zq, q), (epi.zq_t, qt)):
        assert torch.equal(got.data, ref.data) and torch.equal(got.scales, ref.scales)


def test_gelu_chain_over_its_operands(mx):
    """Between four and twelve tiles per SM, where one kernel does it all, codes written over the product's operands still wait for
    all of the product: two kernels, and the results of buffers of their own."""
    M, N = 128 * 148, 512
    _, a, b = operands(mx, M, N, N, 12)
    bufs = [mx.QMat(M, N), mx.QMat(N, M)]
    ys = [torch.empty((M, N), dtype=torch.bfloat16, device="cuda") for _ in range(2)]
    for y, zq, launches in ((ys[0], bufs[0], 1), (ys[1], a, 2)):
        n0 = mx.launch_count()
        mx.gemm_quant(a, b, mx.Epilogue(hook=mx.HOOK_GELU, y=y, zq=zq, zq_t=bufs[1], qp_t=(0, 1, 5, 6), chain=True))
        assert mx.launch_count() == n0 + launches
        if launches == 1:
            want_t = bufs[1].data.clone()
    assert torch.equal(ys[0], ys[1])
    assert torch.equal(a.data, bufs[0].data) and torch.equal(a.scales_linear(), bufs[0].scales_linear()) and torch.equal(bufs[1].data, want_t)


# more tiles than SMs and a short contraction: two groups of epilogue warps, with ragged last tiles.  GELU: 298 tiles (two blocks have a
# third), 171 (23 blocks have a second), 225, 600, contractions of one, two, four and three K tiles.  Multiply: 171, 600 and 4950 tiles, two, three
# and four K tiles (298 and 225 are one group's there, as 4950 is two kernels' behind GELU)
@pytest.mark.parametrize("M,N,K", [(18976, 160, 96), (2400, 1056, 384), (9504, 288, 1024), (12768, 736, 704), (25248, 3104, 992)])
@pytest.mark.parametrize("hook", ["gelu", "multiply"])
def test_two_groups_of_epilogue_warps(mx, M, N, K, hook):
    _, a, b = operands(mx, M, N, K, M + N + K)
    g = torch.Generator(device="cuda").manual_seed(M)
    aux = torch.randn((M, N), generator=g, device="cuda").to(torch.bfloat16)
    bias = torch.randn(N, generator=g, device="cuda").to(torch.bfloat16)
    # Y and Z in pieces, chained and both kept: always one group (held against the oracle above).  The same bits
    y, z = (torch.empty((M, N), dtype=torch.bfloat16, device="cuda") for _ in range(2))
    for r in range(0, M, 1280):
        rows = slice(r, min(r + 1280, M))
        n = rows.stop - r
        part = mx.QMat(n, K, data=a.data[rows].contiguous(), scales=a.scales[r // 128 * ((K // 32 + 3) // 4) * 512:].clone())
        kw = dict(hook=mx.HOOK_GELU) if hook == "gelu" else dict(hook=mx.HOOK_MULTIPLY, aux=aux[rows])
        mx.gemm_quant(part, b, mx.Epilogue(y=y[rows], z=z[rows], zq=mx.QMat(n, N), zq_t=mx.QMat(N, n), chain=True, **kw), bias=bias)
    st = mx.new_status()
    seed = 77 + K
    got_y, got_z = (torch.zeros((M, N), dtype=torch.bfloat16, device="cuda") for _ in range(2))
    if hook == "gelu":
        epi = mx.Epilogue(hook=mx.HOOK_GELU, y=got_y, zq=mx.QMat(M, N), zq_t=mx.QMat(N, M), qp_t=(0, 1, seed, 6), chain=True)
        zq, zq_t = mx.quantize_chain(z, seed)
    else:
        epi = mx.Epilogue(hook=mx.HOOK_MULTIPLY, aux=aux, z=got_z, zq=mx.QMat(M, N), qp_row=(0, 1, seed, 3), zq_t=mx.QMat(N, M), qp_t=(0, 1, seed, 5))
        zq, zq_t = mx.quantize_2axis(z, (0, 1, seed, 3), (0, 1, seed, 5))
    mx.gemm_quant(a, b, epi, bias=bias, dev_status=st)
    torch.cuda.synchronize()
    assert int(st.item()) == 0
    assert torch.equal(got_y, y) if hook == "gelu" else torch.equal(got_z, z)
    for got, want in ((epi.zq, zq), (epi.zq_t, zq_t)):
        assert torch.equal(got.data, want.data) and torch.equal(got.scales, want.scales)


def test_gemm_quant_argument_errors(mx):
    a, b = mx.QMat(128, 64), mx.QMat(128, 64)
    with pytest.raises(mx.MxError) as e:
        mx.gemm_quant(a, b, mx.Epilogue())                       # nothing asked for
    assert e.value.status == 1
    with pytest.raises(mx.MxError) as e:
        mx.gemm_quant(a, b, mx.Epilogue(zq=mx.QMat(128, 128), chain=True))   # a chain needs both results
    assert e.value.status == 1
    with pytest.raises(mx.MxError) as e:
        mx.gemm_quant(a, mx.QMat(72, 64), mx.Epilogue(zq=mx.QMat(128, 72)))  # N must be a multiple of 32
    assert e.value.status == 2


# one tile row (the fused epilogue) and two (two kernels, from four tiles per SM on)
@pytest.mark.parametrize("M", [32, 160])
def test_gelu_of_every_bf16_value(mx, M):
    """Every finite bf16 value as Y.  Z is the rounding to bf16 (2^-8 of the result at most) of a value within 1.1 % of GELU(Y) down to
    2^-125, and within 2e-7 |y|."""
    from scipy.special import erfc
    y = torch.arange(65536, dtype=torch.int32).to(torch.int16).view(torch.bfloat16).cuda()
    y = torch.where(torch.isnan(y), torch.zeros_like(y), y)
    N = y.numel()
    a, b = mx.QMat(M, 32), mx.QMat(N, 32)
    for q in (a, b):
        q.data.zero_()
        q.scales.fill_(127)
    out_y, z = torch.empty((M, N), dtype=torch.bfloat16, device="cuda"), torch.empty((M, N), dtype=torch.bfloat16, device="cuda")
    st = mx.new_status()
    epi = mx.Epilogue(hook=mx.HOOK_GELU, y=out_y, z=z, zq=mx.QMat(M, N), zq_t=mx.QMat(N, M), qp_t=(0, 0, 0, 0), chain=True)
    mx.gemm_quant(a, b, epi, bias=y, dev_status=st)
    torch.cuda.synchronize()
    assert int(st.item()) == mx.DEV_NONFINITE      # of the two infinities
    assert torch.equal(out_y, (y + 0.0).expand(M, N))
    assert torch.equal(z.view(torch.int16), z[:1].view(torch.int16).expand(M, N))
    yv, zv = y.double().cpu().numpy(), z[0].double().cpu().numpy()
    assert zv[yv == np.inf] == np.inf and np.isnan(zv[yv == -np.inf])
    fin = np.isfinite(yv)
    yv, zv = yv[fin], zv[fin]
    want = 0.5 * yv * erfc(-yv * np.sqrt(0.5))
    assert (np.signbit(zv) == (yv < 0)).all()
    assert (np.abs(zv - want) <= np.abs(want) * (2.0 ** -8 + 0.011 * (1 + 2.0 ** -8)) + 2.0 ** -125).all()
    assert (np.abs(zv - want) <= (np.abs(want) + 2e-7 * np.abs(yv)) * 2.0 ** -8 + 2e-7 * np.abs(yv) + 2.0 ** -125).all()
