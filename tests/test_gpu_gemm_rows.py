"""auv_gemm where its dispatch changes kernels: products over many rows with a short contraction (at least 8 row
tiles of 128 and at most 9 K-chunks of 128 bytes), fp32 results stored as boxes where rows and N are whole 16-byte pieces, and tf32
operands read along their samples, in place or, when their rows do not start on 16 bytes, through a copy; and the fp32
CUDA-core kernels (a warp per block, splits in turn, 64- and 128-wide tiles, 16-row tiles, partials in memory), with
16-byte and 4-byte copies.

Against float64 of the same operands; tolerances as in test_gpu_gemm.py, as a fraction of sum_k |A(m,k) B(n,k)|:
fp32 sums of exact bf16 products 1e-5, tf32 operands rounded to nearest (2^-11 each) 3e-3, bf16 results half an ulp."""
import pytest

from parity_util import need_gpu

pytestmark = pytest.mark.gpu
TOL = {"bf16": 1e-5, "tf32": 3e-3, "fp32": 1e-5}


def run(torch, prec, M, N, K, a_mn, b_mn, c_bf16=False, pad_a=0, pad_b=0, pad_c=3, beta=0.0):
    from paper_2512_13359_gb300 import auvenv
    g = torch.Generator(device="cuda").manual_seed(M + 3 * N + 7 * K)
    dt = torch.bfloat16 if prec == "bf16" else torch.float32

    def operand(rows, mn, pad):
        inner, outer = (rows, K) if mn else (K, rows)
        align = {"bf16": 8, "tf32": 4, "fp32": 4}[prec]
        ld = -(-inner // align) * align + pad
        t = torch.randn((outer, ld), generator=g, device="cuda").to(dt)
        v = t[:, :inner].double()
        return t, ld, v.T if mn else v

    A, lda, a = operand(M, a_mn, pad_a)
    B, ldb, b = operand(N, b_mn, pad_b)
    C = torch.full((M, N + pad_c), 7.0, device="cuda", dtype=torch.bfloat16 if c_bf16 else torch.float32)
    ws = torch.empty(auvenv.lib().auv_gemm_workspace_bytes(M, N, K) // 4 + 1, device="cuda")
    if beta:
        C[:, :N] = torch.randn((M, N), generator=g, device="cuda")
    c0 = C[:, :N].double()
    st = auvenv.gemm(prec, M, N, K, A, lda, a_mn, B, ldb, b_mn, C, N + pad_c, beta, ws)
    ref, scale = a @ b.T, a.abs() @ b.abs().T
    if beta:
        ref, scale = ref + beta * c0, scale + abs(beta) * c0.abs()
    tol = TOL[prec] * scale + 1e-30 + (2.0 ** -8 * ref.abs() if c_bf16 else 0.0)
    assert st.cpu().tolist() == [0, 0, 0, 0]
    assert bool(((C[:, :N].double() - ref).abs() <= tol).all())
    assert bool((C[:, N:] == 7.0).all())


@pytest.mark.parametrize("prec", ["bf16", "tf32"])
@pytest.mark.parametrize("M,N,K,b_mn", [
    (1023, 256, 264, False), (1024, 256, 264, False), (1025, 129, 17, True),   # the row line; two 128-wide tiles
    (2000, 64, 288, False), (2000, 64, 289, False), (2000, 64, 576, True), (2000, 64, 577, True),  # chunk lines
    (1100, 8, 1, True)])
def test_short_contractions(prec, M, N, K, b_mn):
    run(need_gpu(), prec, M, N, K, False, b_mn)
    run(need_gpu(), prec, M, N, K, False, b_mn, pad_c=4 + -N % 4)   # 16-byte rows: results stored as boxes


@pytest.mark.parametrize("prec,c_bf16", [("bf16", True), ("bf16", False), ("tf32", False)])
@pytest.mark.parametrize("b_mn", [False, True])
def test_wide_tiles(prec, c_bf16, b_mn):
    torch = need_gpu()
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    for rows in (128 * (sms // 2), 128 * (sms // 2) + 1, 128 * 2 * sms + 5):
        run(torch, prec, rows, 250, 40, False, b_mn, c_bf16)
        run(torch, prec, rows, 252, 40, False, b_mn, c_bf16, pad_c=4)


@pytest.mark.parametrize("prec", ["bf16", "tf32"])
@pytest.mark.parametrize("c_bf16", [False, True])
@pytest.mark.parametrize("N", [16, 33, 128, 255, 256])
@pytest.mark.parametrize("pad_c", [0, 1, 8])
def test_result_added_to_what_is_there(prec, c_bf16, N, pad_c):
    """beta, and rows of C off 16 bytes: columns read and written by a warp together, 8 rows at a time, the last tile 1,
    7, 8 or 9 rows of its warp's 32."""
    for M in (1025, 1024 + 39, 1024 + 72, 1024 + 105):
        for beta in (0.0, -0.5):
            run(need_gpu(), prec, M, N, 40, False, N % 2 == 1, c_bf16, pad_c=pad_c, beta=beta)


@pytest.mark.parametrize("M,N,K", [(256, 264, 5000), (16, 264, 32 * 9 + 1), (130, 24, 33), (1, 1, 1), (33, 290, 700)])
@pytest.mark.parametrize("pad_a,pad_b", [(0, 0), (1, 0), (0, 2), (3, 1)])
def test_tf32_along_samples(M, N, K, pad_a, pad_b):
    run(need_gpu(), "tf32", M, N, K, True, True, False, pad_a, pad_b)
    run(need_gpu(), "tf32", M, N, K, False, True, False, 0, pad_b)
    run(need_gpu(), "tf32", M, N, K, True, False, False, pad_a, 0)


@pytest.mark.parametrize("M,N,K,a_mn", [
    (70, 40, 300, False), (33, 12, 264, False), (1, 1, 9, False),          # a warp per block and split
    (20011, 24, 256, False), (300, 32, 24, False),                         # a warp per block, no split
    (4090, 256, 264, False), (2500, 260, 40, False),                       # 64-wide tiles, splits in turn
    (9800, 256, 24, False), (2003, 250, 17, False), (20000, 250, 264, False),  # 64- and 128-wide tiles
    (40, 50, 2001, False), (12, 264, 5003, True), (16, 100, 24, True), (260, 264, 3000, True), (50, 24, 33, True),
    (17, 70, 4001, True), (32, 264, 3000, False), (33, 130, 3000, True),       # 32-row tiles and one row more
    (2100, 260, 512, False), (2100, 260, 520, False),                          # the splits' chain: in turn, as partials
    (19457, 288, 40, False), (19456, 257, 9, True), (19456, 289, 9, True),     # column tiles of 96
    (128, 128, 128 * 304 * 4, True), (256, 256, 9000, True), (39000, 256, 9, True),   # 128-wide tiles of an MN-major A
    (8000, 1030, 264, False), (8000, 1030, 260, True)])                        # through registers when off 16 bytes
@pytest.mark.parametrize("b_mn", [False, True])
@pytest.mark.parametrize("pad", [0, 1])
def test_fp32_kernels(M, N, K, a_mn, b_mn, pad):
    run(need_gpu(), "fp32", M, N, K, a_mn, b_mn, False, pad, pad, beta=0.5 if M % 2 else 0.0)


@pytest.mark.parametrize("M", [1024, 5000, 40000])
def test_products_that_feed_one_another(M):
    """Launches that overlap the kernel before them: each product reads the
    last one's result (rows kernel, then a contraction over the samples with
    split partials and their reduction, whose result is the next product's
    other operand, in place of one still being read), back to back, one at a
    time, and replayed from a graph: the same bits."""
    torch = need_gpu()
    from paper_2512_13359_gb300 import auvenv
    H = 256
    g = torch.Generator(device="cuda").manual_seed(M)
    x0 = torch.randn((M, H), generator=g, device="cuda")
    w0 = torch.randn((H, H), generator=g, device="cuda") / 16
    x, y, w = (torch.empty_like(t) for t in (x0, x0, w0))
    ws = torch.empty(max(auvenv.lib().auv_gemm_workspace_bytes(m, H, k) for m, k in ((M, H), (H, M))) // 4 + 1,
                     device="cuda")
    st = torch.zeros(4, dtype=torch.int32, device="cuda")

    def chain(sync):
        x.copy_(x0)
        w.copy_(w0)
        for _ in range(6):
            for A, B, C, m, k, mn in ((x, w, y, M, H, False), (y, w, x, M, H, False), (x, y, w, H, M, True)):
                auvenv.gemm("tf32", m, H, k, A, H, mn, B, H, mn, C, H, 0.0, ws, st)
                sync()
            w.mul_(1.0 / w.abs().max() / 16)   # another library's kernel between two of ours
            sync()
        return x.clone(), w.clone()

    one = chain(torch.cuda.synchronize)
    for _ in range(3):
        assert all(torch.equal(a, b) for a, b in zip(one, chain(lambda: None)))
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        out = chain(lambda: None)
    for _ in range(3):
        graph.replay()
        torch.cuda.synchronize()
        assert all(torch.equal(a, b) for a, b in zip(one, out))
    assert st.cpu().tolist() == [0, 0, 0, 0] and bool(torch.isfinite(one[0]).all())
