"""Decoder GEMM through the C ABI against a plain fp32 matrix product of the same bf16 / fp32 inputs."""
import numpy as np
import pytest

from paper_2608_18183_b200 import binding, synth
from tests import gpu_util as G

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx_bf16():
    w = synth.WORKLOADS["tiny_bf16"]
    c = binding.Context(w.shape, G.weights_for(w), 4, 8)
    yield c
    c.hbsjd_destroy()


@pytest.fixture(scope="module")
def ctx_fp32():
    w = synth.WORKLOADS["tiny"]
    c = binding.Context(w.shape, G.weights_for(w), 4, 8)
    yield c
    c.hbsjd_destroy()


@pytest.mark.parametrize("M,N,K", [(128, 128, 64), (128, 64, 128), (64, 32, 64), (200, 384, 128), (1000, 768, 768),
                                   (1024, 2304, 768), (333, 4096, 768), (1024, 768, 2048), (4096, 1024, 2816),
                                   (2048, 16384, 1024), (1, 128, 64), (8192, 3072, 1024), (8192, 1024, 1024),
                                   (5000, 2048, 512), (4999, 5632, 1024), (2304, 16384, 256)])
def test_bf16_gemm_matches_fp32_product(ctx_bf16, M, N, K):
    import torch
    g = torch.Generator(device="cuda").manual_seed(M * 7 + N * 3 + K)
    A = (torch.randn(M, K, generator=g, device="cuda") * 0.5).bfloat16()
    W = (torch.randn(N, K, generator=g, device="cuda") * 0.05).bfloat16()
    C = torch.full((M, N), 7.0, device="cuda", dtype=torch.float32)
    ctx_bf16.hbsjd_gemm(A, W, C)
    ref = A.float() @ W.float().T
    scale = float(ref.abs().max())
    # fp32 accumulation of exact bf16 products: differences are summation-order rounding only
    assert float((C - ref).abs().max()) <= 2e-5 * max(scale, 1.0) * (K / 64) ** 0.5 + 1e-6
    # accumulate mode adds into C
    C0 = torch.randn(M, N, generator=g, device="cuda")
    C1 = C0.clone()
    ctx_bf16.hbsjd_gemm(A, W, C1, accumulate=True)
    assert float((C1 - (C0 + ref)).abs().max()) <= 2e-5 * max(scale, 1.0) * (K / 64) ** 0.5 + 1e-5


def test_bf16_gemm_rows_do_not_depend_on_their_tile(ctx_bf16):
    """A row's result is bit-identical wherever it sits in the batch (what lets Full and Compact
    execution agree bit for bit)."""
    import torch
    g = torch.Generator(device="cuda").manual_seed(5)
    A = torch.randn(512, 768, generator=g, device="cuda").bfloat16()
    W = (torch.randn(768, 768, generator=g, device="cuda") * 0.05).bfloat16()
    C = torch.empty(512, 768, device="cuda")
    ctx_bf16.hbsjd_gemm(A, W, C)
    perm = torch.randperm(512, generator=g, device="cuda")[:77]
    A2 = A[perm].contiguous()
    C2 = torch.empty(77, 768, device="cuda")
    ctx_bf16.hbsjd_gemm(A2, W, C2)
    assert torch.equal(C2, C[perm])


@pytest.mark.parametrize("M,N,K", [(7, 192, 64), (130, 256, 192), (64, 64, 64)])
def test_fp32_gemm(ctx_fp32, M, N, K):
    import torch
    g = torch.Generator(device="cuda").manual_seed(M + N + K)
    A = torch.randn(M, K, generator=g, device="cuda")
    W = torch.randn(N, K, generator=g, device="cuda") * 0.1
    C = torch.zeros(M, N, device="cuda")
    ctx_fp32.hbsjd_gemm(A, W, C)
    ref = (A.double() @ W.double().T).float()
    assert float((C - ref).abs().max()) < 1e-5 * K ** 0.5


def test_bounded_wait_runs_out_and_the_context_recovers(ctx_bf16):
    """The failure path of the GEMM pipeline on a healthy GPU: the epilogue warps' bounded wait for their
    accumulator is shortened to 300 ns while the main loop over K = 8192 needs tens of microseconds, so the wait
    runs out.  The kernel must not hang or fault: it raises its error flag, every role leaves its loop, the copies
    and MMAs in flight are drained, TMEM is freed, and the call returns HBSJD_ETIMEOUT (-5).  The next call on the
    same context runs normally and is correct.  (One CTA per tile: the shape is too small for CTA pairs.)"""
    import torch
    g = torch.Generator(device="cuda").manual_seed(11)
    M, N, K = 256, 256, 8192
    A = (torch.randn(M, K, generator=g, device="cuda") * 0.5).bfloat16()
    W = (torch.randn(N, K, generator=g, device="cuda") * 0.05).bfloat16()
    C = torch.zeros(M, N, device="cuda")
    with pytest.raises(binding.HbsjdError) as e:
        ctx_bf16.hbsjd_debug_gemm(A, W, C, acc_wait_ns=300)
    assert e.value.code == -5
    torch.cuda.synchronize()
    C2 = torch.zeros(M, N, device="cuda")
    ctx_bf16.hbsjd_gemm(A, W, C2)
    ref = A.float() @ W.float().T
    assert float((C2 - ref).abs().max()) <= 2e-5 * max(float(ref.abs().max()), 1.0) * (K / 64) ** 0.5 + 1e-6
    # several launches back to back through the same entry point give the same result as one
    C3 = torch.zeros(M, N, device="cuda")
    ctx_bf16.hbsjd_debug_gemm(A, W, C3, reps=3)
    assert torch.equal(C3, C2)


@pytest.mark.parametrize("tile", [16032, 16064, 32032, 32064])
@pytest.mark.parametrize("M,N,K", [(1, 64, 64), (15, 128, 192), (17, 64, 320), (33, 192, 1088), (128, 1024, 2816),
                                   (301, 576, 1024)])
def test_few_row_kernel_gives_the_tcgen05_kernels_bits(ctx_bf16, tile, M, N, K):
    """The kernel for few rows sums each element's products in the tcgen05 kernel's order: equal bits, whatever the
    remainder of rows and of k-blocks per copy (1, 3, 5, 17, 44 and 16 k-blocks against copies of two or four)."""
    import torch
    g = torch.Generator(device="cuda").manual_seed(M + N + K)
    A = torch.randn(M, K, generator=g, device="cuda").bfloat16()
    W = (torch.randn(N, K, generator=g, device="cuda") * 0.05).bfloat16()
    for acc in (False, True):
        C0 = torch.randn(M, N, generator=g, device="cuda")
        want, got = C0.clone(), C0.clone()
        ctx_bf16.hbsjd_debug_gemm(A, W, want, accumulate=acc, tile=64)
        ctx_bf16.hbsjd_debug_gemm(A, W, got, accumulate=acc, tile=tile)
        assert torch.equal(got, want)


@pytest.mark.parametrize("M,N,K", [(1, 16, 4), (17, 33, 68), (32, 192, 64), (31, 64, 260), (32, 64, 1028), (5, 40, 7),
                                   (304, 496, 64), (320, 496, 64)])
def test_fp32_gemm_small_tiles(ctx_fp32, M, N, K):
    """The 16 x 16 tiles of small fp32 problems: edges of tiles and K panels, more panels than the ring holds, K not a
    multiple of four (the 64 x 64 kernel), and both sides of the largest problem that takes them (19 x 31 tiles = 589,
    20 x 31 = 620 of 4 x 148 = 592).  Bound: K fused multiply-adds, each within half an ulp of the running sum."""
    import torch
    g = torch.Generator(device="cuda").manual_seed(M + N + K)
    A = torch.randn(M, K, generator=g, device="cuda")
    W = torch.randn(N, K, generator=g, device="cuda") * 0.1
    C0 = torch.randn(M, N, generator=g, device="cuda")
    ref = A.double() @ W.double().T
    tol = 2.0 ** -24 * (K + 2) * (A.double().abs() @ W.double().abs().T + C0.abs())
    C = torch.zeros(M, N, device="cuda")
    ctx_fp32.hbsjd_gemm(A, W, C)
    assert bool(((C.double() - ref).abs() <= tol).all())
    C = C0.clone()
    ctx_fp32.hbsjd_gemm(A, W, C, accumulate=True)
    assert bool(((C.double() - C0.double() - ref).abs() <= tol).all())


@pytest.mark.parametrize("tile", [16032, 16064, 32032, 32064])
def test_bounded_wait_of_the_few_row_kernel_runs_out(ctx_bf16, tile):
    """The same failure path in the kernel for few rows: 40 ns are shorter than any copy's way from memory, so the warps
    that wait for their first operands give up, both producers leave and wait for what they have requested, and the
    call returns HBSJD_ETIMEOUT.  The next call is correct."""
    import torch
    g = torch.Generator(device="cuda").manual_seed(tile)
    M, N, K = 40, 256, 8192
    A = (torch.randn(M, K, generator=g, device="cuda") * 0.5).bfloat16()
    W = (torch.randn(N, K, generator=g, device="cuda") * 0.05).bfloat16()
    C = torch.zeros(M, N, device="cuda")
    with pytest.raises(binding.HbsjdError) as e:
        ctx_bf16.hbsjd_debug_gemm(A, W, C, acc_wait_ns=40, tile=tile)
    assert e.value.code == -5
    torch.cuda.synchronize()
    want, got = torch.zeros(M, N, device="cuda"), torch.zeros(M, N, device="cuda")
    ctx_bf16.hbsjd_debug_gemm(A, W, want, tile=64)
    ctx_bf16.hbsjd_debug_gemm(A, W, got, tile=tile)
    assert torch.equal(got, want)


def _wide_operands(kind, M, N, K, g):
    """bf16 operands on which an accumulator that aligned or rounded its products otherwise would show."""
    import torch
    A, W = torch.randn(M, K, generator=g, device="cuda"), torch.randn(N, K, generator=g, device="cuda")
    spread = lambda x, e: x * torch.exp2(((torch.rand(x.shape, generator=g, device="cuda") * 2 - 1) * e).round())
    if kind == "wide":
        A, W = spread(A, 20), spread(W, 20)
    elif kind == "cancelling":  # neighbours cancel, but for the last bit of some
        A, W = spread(A, 10), spread(W, 10)
        A[:, 1::2] = -A[:, 0::2]
        W[:, 1::2] = W[:, 0::2] * (1 + (torch.rand(N, K // 2, generator=g, device="cuda") < 0.3) * 2.0 ** -7)
    elif kind == "running sum":  # a large sum first, products far below its last bits behind it
        A[:, :64] *= 2.0 ** 12
        A[:, 64:] *= 2.0 ** -10
    elif kind == "one large per step":
        big = torch.randn(M, (K + 15) // 16, generator=g, device="cuda") * 2.0 ** 10
        A *= 2.0 ** -14
        A[:, ::16] = big
    elif kind == "denormal":
        A, W = A * 2.0 ** -70, W * 2.0 ** -62
    elif kind == "overflow":
        A, W = A * 2.0 ** 60, W * 2.0 ** 62
    return A.bfloat16().contiguous(), W.bfloat16().contiguous()


@pytest.mark.parametrize("kind", ["wide", "cancelling", "running sum", "one large per step", "denormal", "overflow"])
@pytest.mark.parametrize("M,N,K", [(48, 128, 320), (301, 512, 1024)])
def test_both_gemm_kernels_round_alike(ctx_bf16, kind, M, N, K):
    """mma.sync and tcgen05 sum their 16 products per step alike; no document says so, hence operands of mixed magnitude,
    not random ones of one scale.  Infinities and NaN are compared by their bits too."""
    import torch
    g = torch.Generator(device="cuda").manual_seed(M + K)
    A, W = _wide_operands(kind, M, N, K, g)
    out = []
    for tile in (64, 256, 512, 16032, 16064, 32032, 32064):
        if N % 256 and tile in (256, 512):
            continue
        C = torch.zeros(M, N, device="cuda")
        ctx_bf16.hbsjd_debug_gemm(A, W, C, tile=tile)
        out.append(C.view(torch.int32))
    assert all(torch.equal(out[0], o) for o in out[1:])


@pytest.mark.parametrize("offset", [1, 2, 3])
@pytest.mark.parametrize("M", [8, 600])
def test_output_off_its_16_byte_boundary_is_refused(ctx_bf16, M, offset):
    """A few rows or many: refused on the host, nothing launched."""
    import torch
    A, W = torch.ones(M, 64, device="cuda").bfloat16(), torch.ones(128, 64, device="cuda").bfloat16()
    flat = torch.zeros(M * 128 + 4, device="cuda")
    for accumulate in (False, True):
        with pytest.raises(binding.HbsjdError) as e:
            ctx_bf16.hbsjd_gemm(A, W, flat[offset:offset + M * 128].view(M, 128), accumulate=accumulate)
        assert e.value.code == -1
    assert not bool(flat.any())


@pytest.mark.parametrize("tile", [32, 128, 256, 512])
def test_epilogue_warps_without_rows_leave_the_tile_before_alone(ctx_bf16, tile):
    """4865 rows: the last row of tiles has rows for one warp only, and CTAs come to it from whole tiles while the last of
    those are still being stored (three k-blocks per tile: the main loop is over long before).  The other warps must not
    write into the buffers that these stores read.  Bound: one product's sum in fp32, K = 192, whatever the tile."""
    import torch
    g = torch.Generator(device="cuda").manual_seed(4865)
    A = torch.randn(4865, 192, generator=g, device="cuda").bfloat16()
    W = torch.randn(1024, 192, generator=g, device="cuda").bfloat16()
    ref = A.float() @ W.float().T
    for acc in (True, False) * 3:
        C0 = torch.randn(4865, 1024, generator=g, device="cuda")
        C = C0.clone()
        ctx_bf16.hbsjd_debug_gemm(A, W, C, accumulate=acc, tile=tile)
        assert float((C - (ref + C0 if acc else ref)).abs().max()) < 1e-3


@pytest.mark.parametrize("tile", [96, 160, 192])
@pytest.mark.parametrize("M,K,kind", [(1, 64, "wide"), (17, 192, "cancelling"), (63, 1088, "running sum"), (65, 64, "wide"), (129, 2816, "wide"),
                                      (300, 1280, "cancelling"), (2100, 320, "wide"), (6000, 64, "wide")])
def test_tiles_between_the_powers_of_two(ctx_bf16, tile, M, K, kind):
    """Tiles whose columns are no power of two: edges of rows, 1 to 44 k-blocks against rings of 4 and 6, several tiles per CTA
    (85 to 170 of 2100 rows, 240 of 6000); the 128 x 64 tile's bits."""
    import torch
    N = 960
    g = torch.Generator(device="cuda").manual_seed(M + K)
    A, W = _wide_operands(kind, M, N, K, g)
    for acc in (False, True):
        C0 = torch.randn(M, N, generator=g, device="cuda")
        want, got = C0.clone(), C0.clone()
        ctx_bf16.hbsjd_debug_gemm(A, W, want, accumulate=acc, tile=64)
        ctx_bf16.hbsjd_debug_gemm(A, W, got, accumulate=acc, tile=tile)
        assert torch.equal(got.view(torch.int32), want.view(torch.int32))


@pytest.mark.parametrize("M", [4865, 5120, 7000, 9472, 9473])
def test_last_wave_of_cta_pairs_in_halves(ctx_bf16, M):
    """256 x 256 tiles on 74 CTA pairs, 80, 80, 112, 148 and 152 of them for N = 1024: a rest of 6, 6 and 4 goes as halves, a
    rest of 38 or none whole.  The same bits as one CTA's tiles."""
    import torch
    g = torch.Generator(device="cuda").manual_seed(M)
    A = torch.randn(M, 192, generator=g, device="cuda").bfloat16()
    W = torch.randn(1024, 192, generator=g, device="cuda").bfloat16()
    for acc in (False, True):
        C0 = torch.randn(M, 1024, generator=g, device="cuda")
        want, got = C0.clone(), C0.clone()
        ctx_bf16.hbsjd_debug_gemm(A, W, want, accumulate=acc, tile=128)
        ctx_bf16.hbsjd_debug_gemm(A, W, got, accumulate=acc, tile=512)
        assert torch.equal(got, want)


@pytest.mark.parametrize("M", [300, 2049, 4096])
def test_residual_update_with_norm_sums_on_every_kernel(M):
    """The folded residual update (its bf16 copy and sums of squares come with it) at 1280 columns: tiles of every width that
    one CTA takes, the few-row kernel, and CTA pairs, whose last wave goes as halves at 4096 rows (80 tiles on 74 pairs)
    and whole at 2049 (45 tiles).  The sum is the plain update's; copy and sums of squares are compared through whole
    forwards, in test_every_epilogue_of_cta_pairs_with_a_last_wave_in_halves."""
    import torch
    s = synth.ModelShape(1, 1280, 20, 64, 64, 4, 4, 3, "bf16")
    ctx = binding.Context(s, synth.make_weights(s, 3, target_entropy=None), 64, 32)
    g = torch.Generator(device="cuda").manual_seed(M)
    A = torch.randn(M, 320, generator=g, device="cuda").bfloat16()
    W = torch.randn(1280, 320, generator=g, device="cuda").bfloat16()
    C0 = torch.randn(M, 1280, generator=g, device="cuda")
    want = C0.clone()
    ctx.hbsjd_debug_gemm(A, W, want, accumulate=1, tile=64)
    for tile in (0, 32, 64, 128, 160, 256, 512, 640, 16032, 32064):
        got = C0.clone()
        ctx.hbsjd_debug_gemm(A, W, got, accumulate=2, tile=tile)
        assert torch.equal(got, want), tile
    ctx.hbsjd_destroy()
