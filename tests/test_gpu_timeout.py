"""The drain path of the bounded waits, exercised without any fault.

Every wait on a barrier in the GEMM kernels, the quantizing epilogue and the two-axis quantizer gives up after a bounded number of polls,
raises MXFP4_DEV_TIMEOUT, and makes every role of its thread block leave; the block then frees its tensor memory and
returns.  The self-test entry points launch the real kernels with their loads withheld and the bound at a few
thousand polls, so that path runs within milliseconds: no trap, no endless loop, no bad address.  Afterwards the same
product (and quantizer) must run normally and match the oracle: the tensor memory was handed back and the context is
intact."""
import numpy as np
import pytest
import torch

import oracle as orc
from util import assert_qmat_equal, check_gemm_bound, numpy_to_qmat, to_dev_bf16

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mx():
    import paper_2502_20853_b200 as m
    m.lib()
    assert torch.cuda.is_available()
    return m


def rand_operand(rng, rows, kc):
    c = rng.integers(0, 16, size=(rows, kc)).astype(np.uint8)
    p = (c[:, 0::2] | (c[:, 1::2] << 4)).astype(np.uint8)
    s = rng.integers(122, 132, size=(rows, kc // 32)).astype(np.uint8)
    return p, s


# one shape per kernel of the product: one CTA per tile (128 wide), B-stationary, CTA pairs with split-K, cluster split-K,
# CTA pairs with the B block resident
@pytest.mark.parametrize("M,N,K", [(256, 128, 512), (256, 384, 512), (1024, 512, 2048), (1280, 768, 4096), (4864, 1536, 1024)])
@pytest.mark.parametrize("out_dtype", [0, 1])
def test_gemm_waits_run_out_and_the_kernel_drains(mx, M, N, K, out_dtype):
    rng = np.random.default_rng(M + N + K)
    pa, sa = rand_operand(rng, M, K)
    pb, sb = rand_operand(rng, N, K)
    a, b = numpy_to_qmat(mx, pa, sa), numpy_to_qmat(mx, pb, sb)
    st = mx.new_status()
    mx.gemm_wait_selftest(a, b, st, out_dtype=out_dtype, spin_limit=2048)
    torch.cuda.synchronize()
    assert int(st.item()) & mx.DEV_TIMEOUT, "the withheld loads must make a bounded wait run out"
    # the same kernels, now fed: tensor memory was freed and nothing is left over from the aborted launch
    st.zero_()
    for _ in range(2):
        d = mx.gemm(a, b, out_dtype=out_dtype, dev_status=st)
    torch.cuda.synchronize()
    assert int(st.item()) == 0
    dref, tref = orc.gemm(pa, sa, pb, sb)
    check_gemm_bound(d.float().cpu().numpy(), dref, tref, bf16_out=(out_dtype == 0), what="gemm after the self-test")


# the kernels of products of more than one wave: B-stationary, CTA pairs with and without split K, one CTA per tile
# (192 wide)
@pytest.mark.parametrize("M,N,K", [(9600, 384, 512), (1024, 512, 8192), (9500, 512, 1536), (6272, 512, 1536)])
@pytest.mark.parametrize("out_dtype", [0, 1])
def test_gemm_waits_run_out_beyond_one_wave(mx, M, N, K, out_dtype):
    test_gemm_waits_run_out_and_the_kernel_drains(mx, M, N, K, out_dtype)


def test_quantizer_waits_run_out_and_the_kernel_drains(mx):
    rng = np.random.default_rng(9)
    x = rng.standard_normal((384, 320)).astype(np.float32)
    x = torch.from_numpy(x).to(torch.bfloat16)
    xd = x.cuda()
    st = mx.new_status()
    mx.quantize_wait_selftest(xd, st, spin_limit=2048)
    torch.cuda.synchronize()
    assert int(st.item()) & mx.DEV_TIMEOUT
    st.zero_()
    q, qt = mx.quantize_2axis(xd, (0, 0, 0, 0), (0, 1, 77, 5), dev_status=st)
    torch.cuda.synchronize()
    assert int(st.item()) == 0
    xf = x.float().numpy()
    assert_qmat_equal(q, *orc.quantize(xf)[:2], "row-wise after the self-test")
    assert_qmat_equal(qt, *orc.quantize(xf, transpose=True, rounding=1, seed=77, stream_id=5)[:2], "transposed after the self-test")


def test_selftest_argument_errors(mx):
    a, b = mx.QMat(128, 64), mx.QMat(128, 64)
    with pytest.raises(mx.MxError):
        mx.gemm_wait_selftest(a, b, mx.new_status(), spin_limit=4)          # below the allowed range
    with pytest.raises(mx.MxError):
        mx.gemm_wait_selftest(a, b, None)                                    # the status word is required


@pytest.fixture(scope="module")
def hold():
    """A kernel that lets its successor be placed at once and then takes its time (0.6 s, twice the bound of a wait)."""
    kernel = torch.cuda._compile_kernel(r"""
        extern "C" __global__ void hold(long long ns)
        {
            asm volatile("griddepcontrol.launch_dependents;");
            unsigned long long t0, t;
            asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t0));
            for (int i = 0; i < 2000000; i++) {
                asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
                if ((long long)(t - t0) >= ns) break;
                __nanosleep(1000);
            }
        }""", "hold")
    return lambda: kernel(grid=(1, 1, 1), block=(32, 1, 1), args=[600_000_000])


# one tile per CTA, B-stationary, CTA pairs with split K, cluster split-K, CTA pairs with the B block resident
@pytest.mark.parametrize("M,N,K", [(256, 128, 512), (9600, 384, 512), (1024, 512, 2048), (1280, 768, 4096), (4864, 1536, 1024)])
def test_waits_count_from_the_inputs_on(mx, hold, M, N, K):
    """A product whose blocks are in place long before its inputs exist (behind a slow kernel that lets the quantizer be placed,
    which lets the product be placed) waits for them without its own waits running out."""
    g = torch.Generator(device="cuda").manual_seed(M)
    x = torch.randn((M, K), generator=g, device="cuda").to(torch.bfloat16)
    b = mx.quantize(torch.randn((N, K), generator=g, device="cuda").to(torch.bfloat16))
    a = mx.QMat(M, K)
    st, ws = mx.new_status(), torch.empty(max(mx.gemm_workspace_bytes(M, N, K), 16), dtype=torch.uint8, device="cuda")
    got, want = (torch.full((M, N), float("nan"), dtype=torch.bfloat16, device="cuda") for _ in range(2))
    zq = [mx.QMat(M, N), mx.QMat(M, N)]
    torch.cuda.synchronize()
    for out, z, slow in ((got, zq[0], True), (want, zq[1], False)):
        for product in (lambda: mx.gemm(a, b, out=out, workspace=ws, dev_status=st), lambda: mx.gemm_quant(a, b, mx.Epilogue(zq=z), dev_status=st)):
            if slow:
                a.data.zero_()
                torch.cuda.synchronize()
                hold()
            mx.quantize(x, out=a, dev_status=st)
            product()
            torch.cuda.synchronize()
    assert int(st.item()) == 0
    assert torch.equal(got, want) and torch.equal(zq[0].data, zq[1].data) and torch.equal(zq[0].scales, zq[1].scales)


# the launches of two products: one wave of 128-wide tiles, CTA pairs 256 wide without and with split K, and 192 wide
@pytest.mark.parametrize("M,N,K", [(256, 128, 512), (9600, 512, 1536), (1024, 512, 8192), (384, 384, 8192)])
def test_waits_of_two_products_in_a_launch_run_out(mx, M, N, K):
    """The joint launch of a backward pass drains like a single product's; afterwards a backward pass of the same shapes is right."""
    rng = np.random.default_rng(M)
    a, b = (numpy_to_qmat(mx, *rand_operand(rng, r, K)) for r in (M, N))
    st = mx.new_status()
    before = mx.launch_count()
    mx.gemm_wait_selftest(a, b, st, spin_limit=2048)
    assert mx.launch_count() - before == 2
    torch.cuda.synchronize()
    assert int(st.item()) & mx.DEV_TIMEOUT
    st.zero_()
    # dW [M, N] over K tokens, dX [K, N] over M channels
    dyq_t, xq_t, dyq, wq_t = a, b, numpy_to_qmat(mx, *rand_operand(rng, K, M)), numpy_to_qmat(mx, *rand_operand(rng, N, M))
    ctx = mx.LinearCtx(mx.QMat(K, N), mx.QMat(M, N), xq_t, 7, wq_t)
    dx, dw = mx.linear_bwd(None, ctx, 7, dyq=dyq, dyq_t=dyq_t, dev_status=st)
    torch.cuda.synchronize()
    assert int(st.item()) == 0
    for got, p, q, shape in ((dw, dyq_t, xq_t, (M, N, K)), (dx, dyq, wq_t, (K, N, M))):
        da, db = mx.dequantize(p).double(), mx.dequantize(q).double()
        check_gemm_bound(got.float().cpu().numpy(), (da @ db.T).cpu().numpy(), (da.abs() @ db.abs().T).cpu().numpy(), got.dtype == torch.bfloat16, "after",
                         factor=max(1.0, mx.gemm_chain_mmas(*shape) / 8))


def test_waits_of_two_matrices_in_a_launch_run_out(mx):
    """The forward pass's quantizer of activations and weight drains too (test_quantizer_waits... launches it behind the two-axis one)."""
    x = torch.randn((384, 320), device="cuda").to(torch.bfloat16)
    st = mx.new_status()
    before = mx.launch_count()
    mx.quantize_wait_selftest(x, st, spin_limit=2048)
    assert mx.launch_count() - before == 2
    torch.cuda.synchronize()
    assert int(st.item()) & mx.DEV_TIMEOUT
    st.zero_()
    _, ctx = mx.linear_fwd(x, x, bwd_seed=9, dev_status=st)
    torch.cuda.synchronize()
    assert int(st.item()) == 0
    for got, want in zip((ctx.xq, ctx.xq_t, ctx.wq, ctx.wq_t), mx.quantize_chain(x, seed=9) + mx.quantize_chain(x, seed=9, stream_id_t=4)):
        assert torch.equal(got.data, want.data) and torch.equal(got.scales, want.scales)


# the forward pass of a small batch: clusters of three CTAs, of two, single ones; one and two K tiles
@pytest.mark.parametrize("M,N,K", [(197, 1536, 384), (129, 136, 160), (300, 640, 128)])
def test_waits_of_a_small_forward_pass_run_out(mx, M, N, K):
    g = torch.Generator(device="cuda").manual_seed(M)
    x = torch.randn((M, K), generator=g, device="cuda").to(torch.bfloat16)
    wq = mx.quantize(torch.randn((N, K), generator=g, device="cuda").to(torch.bfloat16))
    want = mx.gemm(mx.quantize(x), wq)
    st = mx.new_status()
    before = mx.launch_count()
    mx.forward_wait_selftest(x, wq, st)
    assert mx.launch_count() - before == 1
    torch.cuda.synchronize()
    assert int(st.item()) & mx.DEV_TIMEOUT
    st.zero_()
    for _ in range(2):
        y, _ = mx.linear_fwd(x, wq=wq, dev_status=st)
    torch.cuda.synchronize()
    assert int(st.item()) == 0 and torch.equal(y, want)


# one group of epilogue warps, and two (171 tiles); with the second factor (a wait of its own) and without
@pytest.mark.parametrize("M,N,K", [(384, 256, 128), (2400, 1056, 384)])
@pytest.mark.parametrize("hook", ["gelu", "multiply"])
def test_waits_of_the_quantizing_epilogue_run_out(mx, M, N, K, hook):
    rng = np.random.default_rng(M)
    a, b = (numpy_to_qmat(mx, *rand_operand(rng, r, K)) for r in (M, N))
    aux = torch.randn((M, N), generator=torch.Generator(device="cuda").manual_seed(N), device="cuda").to(torch.bfloat16)
    y = torch.empty((M, N), dtype=torch.bfloat16, device="cuda")
    q = [mx.QMat(M, N), mx.QMat(N, M)]
    if hook == "gelu":
        epi = mx.Epilogue(hook=mx.HOOK_GELU, y=y, zq=q[0], zq_t=q[1], qp_t=(0, 1, 5, 6), chain=True)
    else:
        epi = mx.Epilogue(hook=mx.HOOK_MULTIPLY, aux=aux, z=y, zq=q[0], qp_row=(0, 1, 5, 3), zq_t=q[1], qp_t=(0, 1, 5, 5))
    st = mx.new_status()
    before = mx.launch_count()
    mx.forward_wait_selftest(a, b, st, epi=epi)
    assert mx.launch_count() - before == 1
    torch.cuda.synchronize()
    assert int(st.item()) & mx.DEV_TIMEOUT
    st.zero_()
    for _ in range(2):
        mx.gemm_quant(a, b, epi, dev_status=st)
    torch.cuda.synchronize()
    assert int(st.item()) == 0
    product = mx.gemm(a, b)
    if hook == "gelu":
        assert torch.equal(y, product) and torch.equal(q[1].data, mx.quantize_t(q[0], rounding=1, seed=5, stream_id=6).data)
    else:
        assert torch.equal(y, product * aux)
        for got, want in zip(q, mx.quantize_2axis(y, (0, 1, 5, 3), (0, 1, 5, 5))):
            assert torch.equal(got.data, want.data) and torch.equal(got.scales, want.scales)


def test_forward_selftest_is_for_one_kernel(mx):
    x, wq, st = torch.ones((128, 512), dtype=torch.bfloat16, device="cuda"), mx.QMat(128, 512), mx.new_status()
    before = mx.launch_count()
    with pytest.raises(mx.MxError):
        mx.forward_wait_selftest(x, wq, st)                                  # two launches
    with pytest.raises(mx.MxError):
        mx.forward_wait_selftest(x[:, :128].contiguous(), mx.QMat(128, 128), st, spin_limit=4)
    assert mx.launch_count() == before


@pytest.mark.parametrize("M,N,K", [(197, 1536, 384), (300, 640, 128)])
def test_waits_of_a_small_forward_pass_count_from_the_inputs_on(mx, hold, M, N, K):
    """Its blocks are in place behind a slow kernel, twice as long as the bound of a wait."""
    x = torch.randn((M, K), device="cuda").to(torch.bfloat16)
    wq = mx.quantize(torch.randn((N, K), device="cuda").to(torch.bfloat16))
    st = mx.new_status()
    want, _ = mx.linear_fwd(x, wq=wq)
    before = mx.launch_count()
    torch.cuda.synchronize()
    hold()
    y, _ = mx.linear_fwd(x, wq=wq, dev_status=st)
    assert mx.launch_count() - before == 1
    torch.cuda.synchronize()
    assert int(st.item()) == 0 and torch.equal(y, want)
