"""GPU parity of the forward pass of a small batch, which quantizes X and multiplies in one launch: codes, scales and product are the
bits of the row-wise quantizer and the product as launches of their own (each held against the oracle elsewhere)."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mx():
    import paper_2502_20853_b200 as m
    m.lib()
    return m


# one row to several row blocks, ragged everywhere; contractions of one group up to the longest, 384; column tiles that divide into
# clusters of 1, 2 and 3 CTAs, one of them in a grid too wide for clusters of three
@pytest.mark.parametrize("M,N,K", [(1, 8, 32), (197, 1536, 384), (31, 384, 96), (128, 1000, 384), (129, 136, 160), (300, 640, 256), (64, 896, 224), (33, 1280, 352),
                                   (2048, 1152, 256), (1792, 1280, 64), (2300, 1024, 320)])
@pytest.mark.parametrize("form", ["plain", "bias_strided_floor"])
def test_forward_in_one_launch(mx, M, N, K, form):
    g = torch.Generator(device="cuda").manual_seed(M + N + K)
    x = torch.randn((M, K + 24), generator=g, device="cuda").to(torch.bfloat16)
    x = x[:, :K] if form != "plain" else x[:, :K].contiguous()
    mode = mx.SCALE_TRUNCATION_FREE if form == "plain" else mx.SCALE_FLOOR
    x[:, : K // 2] *= 0.01
    x[M // 2, -32:] = 0.0
    wq = mx.quantize((torch.randn((N, K), generator=g, device="cuda") * 0.02).to(torch.bfloat16))
    bias = torch.randn(N, generator=g, device="cuda").to(torch.bfloat16) if form != "plain" else None
    st = mx.new_status()
    want_q = mx.quantize(x, scale_mode=mode)
    want = mx.gemm(want_q, wq, bias=bias)
    big = torch.full((M, N + 8), 7.0, dtype=torch.bfloat16, device="cuda")
    n0 = mx.launch_count()
    y, ctx = mx.linear_fwd(x, wq=wq, bias=bias, scale_mode=mode, out=big[:, :N], dev_status=st)
    assert mx.launch_count() == n0 + 1
    torch.cuda.synchronize()
    assert int(st.item()) == 0
    assert torch.equal(y, want) and (big[:, N:] == 7.0).all()
    assert torch.equal(ctx.xq.data, want_q.data) and torch.equal(ctx.xq.scales, want_q.scales)


# on either side of the lines: contractions of 384 and 416, 148 tiles and 149, two CTAs to share the groups of a row block of 384 and one,
# clusters of three in a grid of 126 and pairs and single CTAs in wider ones
@pytest.mark.parametrize("M,N,K,launches", [(40, 1280, 384, 1), (40, 1280, 416, 2), (18944, 96, 64, 1), (18945, 96, 64, 2), (64, 1280, 384, 1),
                                            (64, 640, 384, 2), (64, 640, 256, 1), (1792, 1152, 384, 1), (1800, 1152, 384, 2), (1800, 1152, 224, 1), (1792, 1272, 384, 1)])
def test_lines_of_one_launch(mx, M, N, K, launches):
    g = torch.Generator(device="cuda").manual_seed(M + N + K)
    x = torch.randn((M, K), generator=g, device="cuda").to(torch.bfloat16)
    wq = mx.quantize((torch.randn((N, K), generator=g, device="cuda") * 0.02).to(torch.bfloat16))
    want_q = mx.quantize(x)
    want = mx.gemm(want_q, wq)
    n0 = mx.launch_count()
    y, ctx = mx.linear_fwd(x, wq=wq)
    assert mx.launch_count() == n0 + launches
    assert torch.equal(y, want) and torch.equal(ctx.xq.data, want_q.data) and torch.equal(ctx.xq.scales, want_q.scales)


# Y in the memory of X: as its first columns, at the same address row by row, shifted by rows, and with as many columns; the last three:
# neighbours that share nothing (one launch; the columns beside X lie between its first and last bytes and count as shared)
@pytest.mark.parametrize("M,N,K,x_at,ldx,y_at,ldy,launches", [
    (197, 1536, 384, 0, 1536, 0, 1536, 2), (197, 1536, 384, 0, 384, 0, 1536, 2), (300, 640, 256, 128 * 256, 256, 0, 640, 2), (160, 160, 160, 0, 160, 0, 160, 2),
    (33, 256, 256, 32 * 256 + 248, 256, 0, 256, 2), (197, 1152, 384, 0, 1536, 384, 1536, 2), (197, 1536, 384, 0, 384, 197 * 384, 1536, 1),
    (33, 256, 256, 33 * 256, 256, 0, 256, 1), (33, 256, 96, 32 * 264 + 256, 96, 0, 264, 1)])
def test_y_over_x(mx, M, N, K, x_at, ldx, y_at, ldy, launches):
    g = torch.Generator(device="cuda").manual_seed(M + N)
    size = max(x_at + (M - 1) * ldx + K, y_at + (M - 1) * ldy + N)
    buf = torch.randn(size, generator=g, device="cuda").to(torch.bfloat16)
    x, out = buf.as_strided((M, K), (ldx, 1), x_at), buf.as_strided((M, N), (ldy, 1), y_at)
    wq = mx.quantize((torch.randn((N, K), generator=g, device="cuda") * 0.02).to(torch.bfloat16))
    want, want_ctx = mx.linear_fwd(x.clone(), wq=wq)
    n0 = mx.launch_count()
    y, ctx = mx.linear_fwd(x, wq=wq, out=out)
    assert mx.launch_count() == n0 + launches
    assert torch.equal(y, want)
    assert torch.equal(ctx.xq.data, want_ctx.xq.data) and torch.equal(ctx.xq.scales, want_ctx.xq.scales)


def test_nonfinite_groups_and_a_scale_rule_that_does_not_exist(mx):
    x = torch.ones((40, 128), device="cuda", dtype=torch.bfloat16)
    x[3, 40], x[17, 5] = float("nan"), float("inf")
    wq = mx.quantize(torch.ones((256, 128), device="cuda", dtype=torch.bfloat16))
    st = mx.new_status()
    y, ctx = mx.linear_fwd(x, wq=wq, dev_status=st)
    want = mx.quantize(x)
    torch.cuda.synchronize()
    assert int(st.item()) == mx.DEV_NONFINITE
    assert torch.equal(ctx.xq.data, want.data) and torch.equal(ctx.xq.scales, want.scales)
    bad = torch.isnan(y).any(dim=1).nonzero().flatten().tolist()
    assert bad == [3, 17] and torch.isnan(y[bad]).all()
    n0 = mx.launch_count()
    with pytest.raises(RuntimeError, match="INVALID_ARG"):
        mx.linear_fwd(x, wq=wq, scale_mode=5)
    assert mx.launch_count() == n0


def test_two_launches_in_a_graph(mx):
    x = torch.randn((197, 384), device="cuda").to(torch.bfloat16)
    wq = mx.quantize(torch.randn((1536, 384), device="cuda").to(torch.bfloat16))
    y, ctx = mx.linear_fwd(x, wq=wq)
    torch.cuda.synchronize()
    n0 = mx.launch_count()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        y2, ctx2 = mx.linear_fwd(x, wq=wq)
    assert mx.launch_count() == n0 + 2
    graph.replay()
    torch.cuda.synchronize()
    assert torch.equal(y2, y) and torch.equal(ctx2.xq.data, ctx.xq.data) and torch.equal(ctx2.xq.scales, ctx.xq.scales)
