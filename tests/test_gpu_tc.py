"""Tensor-core ring product (tcgen05 kind::f16 on exact bf16 digit planes)
against the oracle's naive Z_{2^32} triple loop: bit-exact on random,
ragged and adversarial operands.  All digits -128 (a = 0x7F7F7F80) make every
digit product +2^14, so shift group 3 reaches exactly 2^24 at the end of each
256-wide K chunk: the edge of exact fp32 accumulation."""
import numpy as np
import pytest

import oracle as O
from paper_2607_29221_gb300 import workloads as wl
from test_drain_operands import drain_operands

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

ALL_M128 = 0x7F7F7F80      # every signed digit is -128
ALL_P127 = 0x7F7F7F7F      # every signed digit is +127


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2607_29221_gb300 import build
    build.build()
    from paper_2607_29221_gb300 import mosaic as M
    if not M.mosaic_gemm_variant_available(M.GEMM_TC):
        pytest.skip("tensor-core variant not available on this device")
    yield


def _M():
    from paper_2607_29221_gb300 import mosaic as M
    return M


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a).view(np.int32)).cuda()


def host(t):
    torch.cuda.synchronize()
    return t.cpu().numpy().view(np.uint32)


def planes_of(a_dev, rows, K, ldp):
    M = _M()
    p = torch.zeros(4, rows, ldp, dtype=torch.int16, device="cuda")
    if rows and K:
        src = torch.zeros(rows, ldp, dtype=torch.int32, device="cuda")
        src[:, :K] = a_dev
        M.mosaic_digit_split(src, ldp, rows, ldp, p)
    return p


def tc_gemm(A, B):
    M = _M()
    Mm, K = A.shape
    N = B.shape[0]
    ldp = max(8, (K + 7) // 8 * 8)
    Ap = planes_of(dev(A), Mm, K, ldp)
    Bp = planes_of(dev(B), N, K, ldp)
    C = torch.full((Mm, N + 4), -1, dtype=torch.int32, device="cuda")
    M.mosaic_ring_gemm_planes(Ap, ldp, Mm * ldp, Bp, ldp, N * ldp, C, N + 4, Mm, N, K, M.GEMM_TC)
    M.mosaic_device_status()
    got = host(C)
    assert np.all(got[:, N:] == 0xFFFFFFFF)
    return got[:, :N]


def ref(A, B):
    return O.matmul(A, B.T.copy())


@pytest.mark.parametrize("Mm,N,K", [(128, 128, 32), (128, 128, 256), (130, 257, 33), (1, 1, 8),
                                    (300, 129, 1000), (257, 384, 652), (64, 200, 7),
                                    (512, 640, 4096), (129, 1000, 2049)])
def test_tc_random(Mm, N, K):
    A = wl.uniform_u32(11, Mm, K)
    B = wl.uniform_u32(12, N, K)
    assert np.array_equal(tc_gemm(A, B), ref(A, B))


@pytest.mark.parametrize("K", [256, 512, 1024, 768 + 32, 2048])
@pytest.mark.parametrize("va,vb", [(ALL_M128, ALL_M128), (ALL_P127, ALL_M128), (ALL_P127, ALL_P127)])
def test_tc_adversarial_digits(K, va, vb):
    """The largest sums the groups reach (all their terms have one parity here;
    test_tc_drain_points has the sums that would round)."""
    A = np.full((128, K), va, np.uint32)
    B = np.full((128, K), vb, np.uint32)
    assert np.array_equal(tc_gemm(A, B), ref(A, B))


def test_tc_mixed_magnitudes():
    """Large partial sums followed by small products (rounding would drop the small ones)."""
    K = 512
    A = np.full((256, K), ALL_M128, np.uint32)
    B = np.full((128, K), ALL_M128, np.uint32)
    rng = np.random.Generator(np.random.PCG64(5))
    A[:, 200:] = rng.integers(0, 2**32, (256, K - 200), dtype=np.uint64).astype(np.uint32)
    B[::2, 255] = 0x80808081          # digit 0 = +1, others 0
    A[::3, 255] = 0x80808081
    assert np.array_equal(tc_gemm(A, B), ref(A, B))


def test_tc_through_uint32_entry():
    M = _M()
    A = wl.uniform_u32(21, 200, 96)
    B = wl.uniform_u32(22, 300, 96)
    p = M.default_params()
    ws = torch.empty(M.mosaic_workspace_bytes(M.OP_RING_GEMM, 200, 300, 96, p), dtype=torch.uint8,
                     device="cuda")
    C = torch.empty(200, 300, dtype=torch.int32, device="cuda")
    M.mosaic_ring_gemm(dev(A), 96, dev(B), 96, C, 300, 200, 300, 96, M.GEMM_TC, ws)
    M.mosaic_device_status()
    assert np.array_equal(host(C), ref(A, B))


def test_tc_protocol_layer_matches_oracle():
    """The single 64x256x128 layer with the server product on tensor cores."""
    import test_gpu_parity as T
    g, r, op, m, l = T._run_layer(3, (1536, 1024, 652), (80, 80), m=128, n=256, l=64,
                                  variant=_M().GEMM_TC)
    T._check_layer(g, r, op, m, l)


# --------------------------------------------------------------------------
# Few tokens (M <= 16): the TC variant streams uint32 B through TMA instead of
# splitting it into planes; same ring product, checked the same way.
# --------------------------------------------------------------------------
def ring_gemm_u32(A, B, pad_a=0, pad_b=0, variant=None):
    M = _M()
    variant = M.GEMM_TC if variant is None else variant
    Mm, K = A.shape
    N = B.shape[0]
    lda = (K + 3) // 4 * 4 + pad_a
    ldb = (K + 3) // 4 * 4 + pad_b
    Ad = torch.zeros(Mm, lda, dtype=torch.int32, device="cuda")
    Bd = torch.zeros(N, ldb, dtype=torch.int32, device="cuda")
    Ad[:, :K] = dev(A)
    Bd[:, :K] = dev(B)
    C = torch.full((Mm, N + 4), -1, dtype=torch.int32, device="cuda")
    nb = M.mosaic_workspace_bytes(M.OP_RING_GEMM, Mm, N, K)
    ws = torch.empty(max(nb, 16), dtype=torch.uint8, device="cuda")
    M.mosaic_ring_gemm(Ad, lda, Bd, ldb, C, N + 4, Mm, N, K, variant, ws)
    M.mosaic_device_status()
    got = host(C)
    assert np.all(got[:, N:] == 0xFFFFFFFF)
    return got[:, :N]


@pytest.mark.parametrize("Mm", [1, 2, 3, 4, 5, 8, 9, 16])
@pytest.mark.parametrize("N,K", [(1, 1), (61, 128), (59, 129), (300, 652), (1000, 4100), (121, 8192)])
def test_few_tokens_random(Mm, N, K):
    A = wl.uniform_u32(31 + Mm, Mm, K)
    B = wl.uniform_u32(37, N, K)
    assert np.array_equal(ring_gemm_u32(A, B), ref(A, B))


@pytest.mark.parametrize("val", [0xFFFFFFFF, 0x80000000, ALL_M128, ALL_P127])
def test_few_tokens_constant(val):
    """Constant operands: every row of C is K * val^2 mod 2^32 exactly."""
    Mm, N, K = 7, 190, 1000
    A = np.full((Mm, K), val, dtype=np.uint32)
    B = np.full((N, K), val, dtype=np.uint32)
    want = np.uint32((K * val * val) % (1 << 32))
    assert np.all(ring_gemm_u32(A, B) == want)


def test_few_tokens_unaligned_rows():
    """Row strides that are not multiples of 4 words: AUTO takes the CUDA-core
    product, TC refuses them as misaligned."""
    M = _M()
    A = wl.uniform_u32(41, 3, 130)
    B = wl.uniform_u32(42, 77, 130)
    assert np.array_equal(ring_gemm_u32(A, B, pad_a=1, pad_b=3, variant=M.GEMM_AUTO), ref(A, B))
    with pytest.raises(M.MosaicError, match="misaligned"):
        ring_gemm_u32(A, B, pad_a=1, pad_b=3, variant=M.GEMM_TC)


def test_few_tokens_edges():
    """17 tokens leave the streaming kernel; K = 0 gives zeros."""
    A = wl.uniform_u32(43, 17, 300)
    B = wl.uniform_u32(44, 65, 300)
    assert np.array_equal(ring_gemm_u32(A, B), ref(A, B))
    M = _M()
    C = torch.full((2, 8), -1, dtype=torch.int32, device="cuda")
    Z = torch.zeros(2, 4, dtype=torch.int32, device="cuda")
    M.mosaic_ring_gemm(Z, 4, Z, 4, C, 8, 2, 2, 0, M.GEMM_TC)
    got = host(C)
    assert np.all(got[:, :2] == 0) and np.all(got[:, 2:] == 0xFFFFFFFF)


# --------------------------------------------------------------------------
# 17..64 tokens: the TC variant streams uint32 B by TMA, splits it into fp16
# digits in tensor memory on the chip and runs 4 MMAs per 16 K (one per digit
# of B, N = (4 - i) x token tile); stream-K over (128-row tile, 256-K chunk)
# units, partial tiles added with red.add.
# --------------------------------------------------------------------------
@pytest.mark.parametrize("Mm", [17, 24, 32, 33, 48, 49, 64])
@pytest.mark.parametrize("N,K", [(1, 1), (61, 128), (129, 33), (300, 652), (1000, 4100), (121, 8192),
                                 (257, 257)])
def test_streamw_tokens_random(Mm, N, K):
    A = wl.uniform_u32(131 + Mm, Mm, K)
    B = wl.uniform_u32(137, N, K)
    assert np.array_equal(ring_gemm_u32(A, B), ref(A, B))


@pytest.mark.parametrize("Mm", [20, 40, 64])
@pytest.mark.parametrize("va,vb", [(ALL_M128, ALL_M128), (ALL_P127, ALL_M128), (0xFFFFFFFF, 0x80000000),
                                   (0xFFFFFFFF, 0xFFFFFFFF)])
def test_streamw_tokens_adversarial(Mm, va, vb):
    """Constant digits over K = 3000: shift group 3 reaches 2^24 at every drain
    with all digits -128; every entry is K va vb mod 2^32."""
    Mm, N, K = Mm, 300, 3000
    A = np.full((Mm, K), va, np.uint32)
    B = np.full((N, K), vb, np.uint32)
    want = np.uint32((K * va * vb) % (1 << 32))
    assert np.all(ring_gemm_u32(A, B) == want)


def test_streamw_tokens_many_tiles_and_units():
    """More (tile, chunk) units than SMs with a ragged last tile and K chunk:
    CTAs start and end inside tiles."""
    A = wl.uniform_u32(141, 40, 5000)
    B = wl.uniform_u32(142, 20000 + 77, 5000)
    assert np.array_equal(ring_gemm_u32(A, B), ref(A, B))


@pytest.mark.parametrize("N", [5000, 9984])
def test_tc_whole_waves_then_stream_k(N):
    """160 (312) tiles on 152 SMs with 8 K chunks: the first one (two) waves of
    tiles run whole, one tile per CTA per wave, and the last 8 tiles' chunks
    are shared by all CTAs."""
    A = wl.uniform_u32(51, 512, 2048)
    B = wl.uniform_u32(52, N, 2048)
    assert np.array_equal(tc_gemm(A, B), ref(A, B))



# --------------------------------------------------------------------------
# Legacy mma.sync s8 variant (int8 digit planes, int32 accumulators)
# --------------------------------------------------------------------------
@pytest.mark.parametrize("Mm,N,K", [(1, 1, 1), (64, 64, 64), (65, 130, 33), (300, 129, 1000), (128, 257, 2049),
                                    (17, 999, 4096)])
def test_mma_s8_random(Mm, N, K):
    M = _M()
    if not M.mosaic_gemm_variant_available(M.GEMM_MMA_S8):
        pytest.skip("mma.sync s8 variant not available")
    A = wl.uniform_u32(61, Mm, K)
    B = wl.uniform_u32(62, N, K)
    assert np.array_equal(ring_gemm_u32(A, B, variant=M.GEMM_MMA_S8), ref(A, B))


@pytest.mark.parametrize("va,vb", [(ALL_M128, ALL_M128), (ALL_P127, ALL_M128), (0xFFFFFFFF, 0x80000000)])
def test_mma_s8_adversarial(va, vb):
    """Constant digits over K = 5000: the int32 group sums wrap mod 2^32."""
    M = _M()
    if not M.mosaic_gemm_variant_available(M.GEMM_MMA_S8):
        pytest.skip("mma.sync s8 variant not available")
    Mm, N, K = 70, 90, 5000
    A = np.full((Mm, K), va, np.uint32)
    B = np.full((N, K), vb, np.uint32)
    want = np.uint32((K * va * vb) % (1 << 32))
    assert np.all(ring_gemm_u32(A, B, variant=M.GEMM_MMA_S8) == want)


@pytest.mark.parametrize("Mm", [8, 9, 13, 16])
@pytest.mark.parametrize("N,K", [(300, 652), (20000 + 77, 1100)])
def test_few_tokens_with_and_without_workspace(Mm, N, K):
    """9 to 16 tokens stream B through the tensor cores when `ws` holds A's
    planes and B is not small (here 20077 rows), through the CUDA cores
    otherwise; 17 need the room."""
    M = _M()
    A = wl.uniform_u32(151 + Mm, Mm, K)
    B = wl.uniform_u32(152, N, K)
    want = ref(A, B)
    assert np.array_equal(ring_gemm_u32(A, B), want)
    C = torch.full((17, N), -1, dtype=torch.int32, device="cuda")
    Ad = torch.from_numpy(np.vstack([A] * 3)[:17].view(np.int32)).cuda()
    Bd = torch.from_numpy(B.view(np.int32)).cuda()
    for ws in (None, torch.empty(8 * Mm * K - 512, dtype=torch.uint8, device="cuda")):
        M.mosaic_ring_gemm(Ad, K, Bd, K, C, N, Mm, N, K, M.GEMM_TC, ws)
        M.mosaic_device_status()
        assert np.array_equal(host(C)[:Mm], want)
    with pytest.raises(M.MosaicError, match="workspace"):
        M.mosaic_ring_gemm(Ad, K, Bd, K, C, N, 17, N, K, M.GEMM_TC, None)


@pytest.mark.parametrize("Mm", [1, 3, 8, 11])
@pytest.mark.parametrize("N", [31, 4560, 4561, 6841, 7000, 9120, 9121, 11404, 18241])
def test_few_tokens_tile_heights(Mm, N):
    """One wave of 30-row tiles, and one to three waves of tiles cut to fill them
    evenly (31 to 60 rows: some warps have a row less than others, the last tile
    is ragged); no workspace, so the CUDA-core kernel runs."""
    M = _M()
    K = 260
    A = wl.uniform_u32(161 + Mm, Mm, K)
    B = wl.uniform_u32(162, N, K)
    C = torch.full((Mm, N), -1, dtype=torch.int32, device="cuda")
    M.mosaic_ring_gemm(torch.from_numpy(A.view(np.int32)).cuda(), K, torch.from_numpy(B.view(np.int32)).cuda(), K, C,
                       N, Mm, N, K, M.GEMM_TC, None)
    M.mosaic_device_status()
    assert np.array_equal(host(C), ref(A, B))


# Few tiles of 2 to 5 chunks: K is split over idle SMs where that saves two chunks or more (one tile;
# 50 and 51 tiles of 3 chunks, on both sides of a second chunk per CTA), ragged rows and K tails.
@pytest.mark.parametrize("Mm,N,K", [(65, 130, 652), (100, 128, 513), (70, 6400, 652), (70, 6401, 652), (300, 700, 1100),
                                    (129, 3000, 1030), (65, 256, 300)])
def test_tc_few_tiles_split_k(Mm, N, K):
    A = wl.uniform_u32(171, Mm, K)
    B = wl.uniform_u32(172, N, K)
    assert np.array_equal(ring_gemm_u32(A, B), ref(A, B))


@pytest.mark.parametrize("Mm,N", [(128, 128), (1600, 1500)])
@pytest.mark.parametrize("stages", [1, 4, 5, 8, 9, 12, 13, 16, 17, 20, 21, 24, 25, 28, 29, 33, 45])
def test_tc_drain_points(Mm, N, stages):
    """Every place of the two drains in a tile's last chunk (K of 1 to 45 stages
    of 32), one tile shared by CTAs and whole tiles one after another, with
    operands whose sums leave fp32's integers when a pair of shift groups is
    kept one stage too long (tests/test_drain_operands.py)."""
    for K in (32 * stages, 32 * stages - 27):
        A, B, S = drain_operands(Mm, N, K)
        want = ref(A[:S], B[:S])[np.ix_(np.arange(Mm) % S, np.arange(N) % S)]
        assert np.array_equal(tc_gemm(A, B), want), K
