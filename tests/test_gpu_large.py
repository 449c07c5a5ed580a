"""The largest sizes: a gradient-shaped tensor with more than 2^32 elements (the stochastic-rounding counters pass
2^32, every offset needs 64 bits, the token count is not a multiple of 128) through the two-axis quantizer, and the
product with a small weight.  Checked on sampled rows / slabs that the oracle computes by itself."""
import numpy as np
import pytest
import torch

import oracle as orc
from util import check_gemm_bound

pytestmark = pytest.mark.gpu

ROWS, COLS = (1 << 20) + 160, 4096          # 4.295e9 elements; 1048736 = 8193 * 128 + 32


@pytest.fixture(scope="module")
def mx():
    import paper_2502_20853_b200 as m
    m.lib()
    assert torch.cuda.is_available()
    return m


@pytest.fixture(scope="module")
def big(mx):
    free, _ = torch.cuda.mem_get_info()
    if free < 24 << 30:
        pytest.skip("needs 24 GB of free device memory")
    g = torch.Generator(device="cuda").manual_seed(20853)
    x = torch.empty((ROWS, COLS), dtype=torch.bfloat16, device="cuda")
    step = 1 << 16
    for r in range(0, ROWS, step):          # heavy-tailed small values, like a gradient
        n = min(step, ROWS - r)
        t = torch.randn((n, COLS), device="cuda", generator=g) * torch.exp(torch.randn((n, 1), device="cuda", generator=g))
        x[r:r + n] = (t * 1e-3).to(torch.bfloat16)
    seed = 0x5EED0000 + 77
    st = mx.new_status()
    q, qt = mx.quantize_2axis(x, (0, 1, seed, 3), (0, 1, seed, 5), dev_status=st)
    torch.cuda.synchronize()
    assert int(st.item()) == 0
    yield x, q, qt, seed
    del x, q, qt
    torch.cuda.empty_cache()


def rows_of(t, idx, as_float=False):
    sel = t[torch.as_tensor(idx, device=t.device)]
    return (sel.float() if as_float else sel).cpu().numpy()


def test_rowwise_operand_beyond_2_to_32_elements(mx, big):
    x, q, qt, seed = big
    rng = np.random.default_rng(1)
    rows = sorted(set(rng.integers(0, ROWS, 12).tolist()) | {0, ROWS - 1, ROWS - 33, (1 << 20) - 1, 1 << 20})
    xs = rows_of(x, rows, as_float=True)
    p = rows_of(q.data, rows)
    s = rows_of(q.scales_linear(), rows)
    for k, r in enumerate(rows):
        pr, sr, _ = orc.quantize(np.ascontiguousarray(xs[k:k + 1]), rounding=1, seed=seed, stream_id=3, out_row0=int(r), out_ld=COLS)
        assert (s[k] == sr[0]).all(), "scales of row %d" % r
        assert (p[k] == pr[0]).all(), "codes of row %d" % r


def test_transposed_operand_beyond_2_to_32_elements(mx, big):
    x, q, qt, seed = big
    # 32-row groups x 32-column blocks; the last column block with late rows has output indices above 2^32
    for r0, c0 in [(0, 0), (ROWS - 32, COLS - 32), (1 << 20, COLS - 32), (524288, 2048), (ROWS - 160, 32)]:
        sub = x[r0:r0 + 32, c0:c0 + 32].float().cpu().numpy()
        ps, ss, _ = orc.quantize(np.ascontiguousarray(sub), transpose=True, rounding=1, seed=seed, stream_id=5,
                                 out_row0=int(c0), out_col0=int(r0), out_ld=ROWS)
        gp = qt.data[c0:c0 + 32, r0 // 2:r0 // 2 + 16].cpu().numpy()
        gs = qt.scales_linear()[c0:c0 + 32, r0 // 32].cpu().numpy()
        assert (gs == ss[:, 0]).all(), "scales at rows %d, cols %d" % (r0, c0)
        assert (gp == ps).all(), "codes at rows %d, cols %d" % (r0, c0)
    assert (COLS - 1) * ROWS + ROWS - 1 >= 1 << 32     # the last slab's output indices pass 2^32


def test_product_with_8194_row_tiles(mx, big):
    x, q, qt, seed = big
    n = 256
    g = torch.Generator(device="cuda").manual_seed(5)
    w = (torch.randn((n, COLS), device="cuda", generator=g) * 0.02).to(torch.bfloat16)
    wq = mx.quantize(w)
    st = mx.new_status()
    y = mx.gemm(q, wq, dev_status=st)
    torch.cuda.synchronize()
    assert int(st.item()) == 0
    rng = np.random.default_rng(2)
    rows = sorted(set(rng.integers(0, ROWS, 20).tolist()) | {0, 127, 128, ROWS - 1, ROWS - 32, ROWS - 33})
    pa, sa = rows_of(q.data, rows), rows_of(q.scales_linear(), rows)
    pb, sb = wq.data.cpu().numpy(), wq.scales_linear().cpu().numpy()
    dref, tref = orc.gemm(pa, sa, pb, sb)
    check_gemm_bound(rows_of(y, rows, as_float=True), dref, tref, True, "Y on sampled rows of 1048736")


def test_quantizing_epilogue_beyond_2_to_36_elements(mx):
    """Outputs with more than 2^36 elements: the random counters (one per 16 elements) pass 2^32 and take the quantizer's
    passes through their wide-counter form, along the rows and along the columns."""
    M, N, K = (1 << 23) + 160, 8224, 32
    assert M * N > 1 << 36
    torch.cuda.empty_cache()
    free, _ = torch.cuda.mem_get_info()
    if free < 84 << 30:
        pytest.skip("needs 84 GB of free device memory")
    g = torch.Generator(device="cuda").manual_seed(36)
    a = mx.quantize(torch.randn((M, K), device="cuda", generator=g).to(torch.bfloat16))
    b = mx.quantize(torch.randn((N, K), device="cuda", generator=g).to(torch.bfloat16))
    new = lambda r, c: mx.QMat(r, c, data=torch.empty((r, c // 2), dtype=torch.uint8, device="cuda"),  # noqa: E731
                               scales=torch.empty(mx.scale_bytes(r, c), dtype=torch.uint8, device="cuda"))
    zq, zq_t = new(M, N), new(N, M)
    st, seed = mx.new_status(), 0x5EED0000 + 36
    mx.gemm_quant(a, b, mx.Epilogue(zq=zq, qp_row=(0, 1, seed, 3), zq_t=zq_t, qp_t=(0, 1, seed, 5)), dev_status=st)
    torch.cuda.synchronize()
    assert int(st.item()) == 0
    bf = mx.dequantize(b)
    for r0, c0 in [(0, 0), (M - 32, N - 32), (M - 32, 0), (M - 192, N - 64)]:
        rows = torch.arange(r0, r0 + 32, device="cuda")
        sa = torch.stack([a.scales[mx.scale_offset(r, 0, K)] for r in range(r0, r0 + 32)])
        codes = a.data[rows].cpu().numpy()
        z = torch.from_numpy(orc.dequantize(codes, sa.cpu().numpy().reshape(32, 1))).cuda().double() @ bf[c0:c0 + 32].double().t()
        z = z.to(torch.bfloat16).float().cpu().numpy()          # 32 exact products per element: one rounding
        p, s, _ = orc.quantize(z, rounding=1, seed=seed, stream_id=3, out_row0=r0, out_col0=c0, out_ld=N)
        got = torch.stack([zq.scales[mx.scale_offset(r, c0 // 32, N)] for r in range(r0, r0 + 32)]).cpu().numpy()
        assert (got == s[:, 0]).all() and (zq.data[rows, c0 // 2:c0 // 2 + 16].cpu().numpy() == p).all(), (r0, c0)
        p, s, _ = orc.quantize(z, transpose=True, rounding=1, seed=seed, stream_id=5, out_row0=c0, out_col0=r0, out_ld=M)
        got = torch.stack([zq_t.scales[mx.scale_offset(c, r0 // 32, M)] for c in range(c0, c0 + 32)]).cpu().numpy()
        assert (got == s[:, 0]).all() and (zq_t.data[c0:c0 + 32, r0 // 2:r0 // 2 + 16].cpu().numpy() == p).all(), (r0, c0)
    del zq, zq_t, a
    torch.cuda.empty_cache()
