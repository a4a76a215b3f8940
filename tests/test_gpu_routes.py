"""Which kernels a call runs on both sides of each dispatch line (where the other
side is the faster one), and that the result does not depend on it: random
operands against the CUDA-core variant or another form of the same call."""
import numpy as np
import pytest

from paper_2607_29221_gb300 import workloads as wl

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


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


def M_():
    from paper_2607_29221_gb300 import mosaic as M
    return M


def sms():
    return torch.cuda.get_device_properties(0).multi_processor_count


def u32(seed, *shape):
    return torch.from_numpy(wl.uniform_u32(seed, *shape).view(np.int32)).cuda()


def empty(*shape):
    return torch.empty(*shape, dtype=torch.int32, device="cuda")


def ws(nbytes):
    return torch.empty(max(int(nbytes), 256), dtype=torch.uint8, device="cuda")


# Few tokens: the streaming kernel below K = 1024 while its 60-row tiles are one wave, tensor cores beyond.
@pytest.mark.parametrize("m", [9, 16])
@pytest.mark.parametrize("waves,dn,K,streamed", [(0, 64, 64, False), (0, 300, 1020, False), (0, 33, 1024, True),
                                                 (1, 0, 256, False), (1, 1, 256, True), (2, 5, 36, True)])
def test_product_of_9_to_16_tokens(kernels, m, waves, dn, K, streamed):
    M = M_()
    N = waves * 60 * sms() + dn
    A, B, C, want = u32(1, m, K), u32(2, N, K), empty(m, N), empty(m, N)
    w = ws(M.mosaic_workspace_bytes(M.OP_RING_GEMM, m, N, K))
    names = kernels(lambda: M.mosaic_ring_gemm(A, K, B, K, C, N, m, N, K, M.GEMM_AUTO, w))
    assert names == ({"split_f16_start", "ring_gemm_tcw"} if streamed else {"ring_gemm_skinny"})
    M.mosaic_ring_gemm(A, K, B, K, want, N, m, N, K, M.GEMM_IMAD)
    assert torch.equal(C, want)


# The check: one launch of clusters while their blocks are all resident at once (about 2400 tokens of up to 4
# vectors, 1200 of more, twice that with many columns), streaming products beyond, where the strides allow them.
@pytest.mark.parametrize("k,l,m,n,dz,clusters", [
    (4, 600, 300, 64, 0, True), (4, 5000, 64, 64, 0, False), (3, 5000, 64, 64, 1, True), (16, 1000, 64, 32, 0, True),
    (16, 2000, 64, 32, 0, False), (9, 2000, 1024, 1024, 0, True), (8, 5000, 1024, 1024, 0, False)])
def test_check_of_many_tokens(kernels, k, l, m, n, dz, clusters):
    M = M_()
    a, Yc, Z, X = (wl.uniform_u32(i, *s) for i, s in enumerate(((k, m), (k, n), (l, m + dz), (l, n))))
    a[:, :k] = np.eye(k, dtype=np.uint32)
    Z[:, :k] = X @ Yc.T - Z[:, k:m] @ a[:, k:].T    # honest answers, then every 7th token is tampered with
    Z[::7, m - 1] += np.uint32(1)                   # an error of 1 shows in every vector whose last entry is not 0
    want = np.count_nonzero(Z[:, :m] @ a.T != X @ Yc.T, axis=1)
    dev = lambda x: torch.from_numpy(x.view(np.int32)).cuda()
    bad, n_bad = empty(l), torch.zeros(1, dtype=torch.int32, device="cuda")
    w = ws(M.mosaic_workspace_bytes(M.OP_FREIVALDS_CHECK, k, 0, l))
    args = [dev(x) for x in (a, Yc, Z, X)]
    names = kernels(lambda: M.mosaic_freivalds_check(k, args[0], args[1], m, n, l, args[2], m + dz, args[3], n, bad,
                                                     n_bad, w))
    assert names == ({"freivalds_check"} if clusters else {"ring_gemm_skinny", "freivalds_compare"})
    assert np.array_equal(bad.cpu().numpy(), want)
    assert int(n_bad) == np.count_nonzero(want) > 0


# The one-launch unmask of up to 16 tokens and the general path (a product that streams L, then gathers) on both sides
# of each line; `rows` counts rounds of one row a warp (152 SMs x 16 warps). ldz = m + sum(r) + pad.
@pytest.mark.parametrize("l,r,t,rounds,dm,pad,few", [
    (1, (4096,), (), 0, 4096, 0, True), (2, (4096,), (), 0, 8192, 0, False), (1, (256,), (), 10, 0, 0, True),
    (1, (256,), (), 10, 4, 0, False), (2, (96, 64, 8192), (8, 4), 0, 4096, 0, False), (2, (96, 64, 4096), (8, 4), 0, 8192, 0, True),
    (4, (8196,), (), 1, 0, 0, True), (3, (8196,), (), 1, 4, 0, False), (4, (8192,), (), 1, 4, 0, True),
    (8, (2052,), (), 1, 0, 0, True), (5, (2052,), (), 1, 4, 0, False), (8, (2052,), (), 2, 0, 1, True),
    (8, (2048,), (), 2, 0, 0, True), (8, (2052,), (), 2, 4, 0, True), (8, (96, 2052), (40,), 2, 0, 0, True),
    (8, (1796,), (), 5, 0, 0, False), (8, (1792,), (), 5, 0, 0, True), (8, (1796,), (), 7, 0, 0, True),
    (8, (3072,), (), 4, 4, 0, True), (8, (3076,), (), 4, 4, 0, False),
    (16, (1600,), (), 1, 0, 0, True), (9, (1604,), (), 1, 0, 0, False), (9, (1280,), (), 0, 124, 0, True),
    (16, (1284,), (), 0, 124, 0, False), (16, (64, 1300), (4,), 1, 0, 0, True), (16, (64, 1304), (4,), 1, 0, 0, False),
    (12, (848,), (), 1, 4, 0, True), (16, (856,), (), 2, 0, 0, False), (16, (64, 856), (4,), 2, 0, 0, True),
    (9, (1600,), (), 2, 4, 0, True), (16, (1604,), (), 2, 4, 0, False), (16, (64, 1360), (4,), 2, 4, 0, True),
    (16, (64, 1364), (4,), 2, 4, 0, False), (16, (64, 2000), (5,), 2, 4, 0, True)])
def test_unmask_of_few_tokens(kernels, l, r, t, rounds, dm, pad, few):
    M = M_()
    m, d, S = rounds * 16 * sms() + dm, len(r), sum(r)
    p = M.default_params(d=d, r=r, t=(0,) + t)
    g = torch.Generator(device="cuda").manual_seed(1)
    rand = lambda *s: torch.randint(-(1 << 31), 1 << 31, s, generator=g, device="cuda", dtype=torch.int64).to(torch.int32)
    ldz = m + S + (4 - (m + S)) % 4 + pad
    Z, K, L, s_w, s_x = rand(l, ldz), rand(l, m), rand(m, r[-1]), torch.rand(m, device="cuda"), torch.rand(l, device="cuda")
    S_idx = torch.cat([rand(m * t[i]).abs() % r[i] for i in range(d - 1)]) if t else None
    S_val = rand(m * sum(t)) if t else None
    w = ws(M.mosaic_workspace_bytes(M.OP_UNMASK, m, 0, l, p))
    out = {v: (torch.empty(l, m, device="cuda"), empty(l, m)) for v in (M.GEMM_AUTO, M.GEMM_IMAD)}
    call = lambda v: M.mosaic_unmask(p, l, m, Z, ldz, K, L, S_idx, S_val, s_w, s_x, None, *out[v], m, v, w)
    names = kernels(lambda: call(M.GEMM_AUTO))
    if few:
        assert names == {"unmask_few"}
    else:
        assert "unmask_few" not in names and ("ring_gemm_skinny" if l <= 8 else "ring_gemm_tcw") in names
    call(M.GEMM_IMAD)
    assert all(torch.equal(a, b) for a, b in zip(out[M.GEMM_AUTO], out[M.GEMM_IMAD]))


# Direct and staged gathers on both sides of each line, for Init X (images of C and J prepared) and the unmask: one
# (entity, 32-row tile) pair a warp (152 SMs x 32), 8192 pairs with two levels of short lists, 40 or 48 entities.
@pytest.mark.parametrize("r,t,n_pad,m,l,direct", [
    ((96, 64, 40), (8, 4), 1024, 1056, 126, True), ((96, 64, 40), (8, 4), 1024, 1056, 127, False),
    ((200, 180, 40), (80, 84), 1024, 1408, 64, True), ((200, 180, 40), (80, 84), 1024, 1408, 65, False),
    ((64, 40), (12,), 512, 1920, 64, True), ((64, 40), (12,), 512, 1920, 65, False), ((64, 40), (8,), 512, 1920, 65, True),
    ((64, 40), (12,), 8192, 20000, 48, True), ((64, 40), (12,), 8192, 20000, 49, False),
    ((64, 40), (16,), 8192, 20000, 40, True), ((64, 40), (16,), 8192, 20000, 41, False),
    ((256, 40), (32,), 8192, 20000, 48, True), ((64, 40), (16,), 8192, 13632, 48, True),
    ((64, 40), (16,), 8192, 13696, 48, False), ((64, 40), (16,), 8192, 13632, 49, False)])
def test_init_x_gathers(kernels, r, t, n_pad, m, l, direct):
    M = M_()
    p, S = M.default_params(d=len(r), r=r, t=(0,) + t), sum(r)
    key = M.make_key(wl.mask_key())
    C, J = u32(1, n_pad, S), u32(2, m, S)
    cj = ws(M.mosaic_workspace_bytes(M.OP_ACTIVATION_PLANES, m, n_pad, 0, p)).view(torch.int16)
    M.mosaic_prepare_activation(p, m, n_pad, C, J, cj)
    w = ws(M.mosaic_workspace_bytes(M.OP_MASK_ACTIVATION, m, n_pad, l, p))
    out = [[empty(l, n_pad), empty(l, m)] for _ in range(2)]
    names = kernels(lambda: M.mosaic_mask_activation_planes(p, key, 9, m, n_pad, l, C, J, cj, *out[0], M.GEMM_AUTO, w))
    assert ("dgather" in names, "pgather" in names) == (direct, not direct)
    M.mosaic_mask_activation(p, key, 9, m, n_pad, l, C, J, *out[1], M.GEMM_IMAD, w)   # no images: staged
    assert all(torch.equal(a, b) for a, b in zip(*out))


@pytest.mark.parametrize("r,t,l,m,direct", [
    ((96, 64, 40), (8, 4), 96, 2730, True), ((96, 64, 40), (8, 4), 96, 2731, False),
    ((200, 180, 40), (80, 84), 64, 2432, True), ((200, 180, 40), (80, 84), 64, 2433, False),
    ((64, 40), (12,), 20, 4864, True), ((64, 40), (12,), 20, 4865, False), ((64, 40), (8,), 20, 4865, True)])
def test_unmask_gathers(kernels, r, t, l, m, direct):
    M = M_()
    p, S, d = M.default_params(d=len(r), r=r, t=(0,) + t), sum(r), len(r)
    Z, K, L, s_w, s_x = u32(1, l, m + S), u32(2, l, m), u32(3, m, r[-1]), torch.rand(m).cuda(), torch.rand(l).cuda()
    S_idx = torch.cat([torch.randint(0, r[i], (m * t[i],), dtype=torch.int32) for i in range(d - 1)]).cuda()
    S_val = u32(4, m, sum(t))
    Lp = ws(M.mosaic_workspace_bytes(M.OP_UNMASK_PLANES, m, 0, 0, p)).view(torch.int16)
    M.mosaic_prepare_unmask(p, m, L, Lp)
    w = ws(M.mosaic_workspace_bytes(M.OP_UNMASK, m, 0, l, p))
    out = {v: (torch.empty(l, m, device="cuda"), empty(l, m)) for v in (M.GEMM_AUTO, M.GEMM_IMAD)}
    call = lambda v: M.mosaic_unmask_planes(p, l, m, Z, m + S, K, L, Lp, S_idx, S_val, s_w, s_x, None, *out[v], m, v, w)
    names = kernels(lambda: call(M.GEMM_AUTO))
    assert ("dgather" in names, "pgather" in names) == (direct, not direct)
    assert "dgather" not in kernels(lambda: call(M.GEMM_IMAD))
    assert all(torch.equal(a, b) for a, b in zip(out[M.GEMM_AUTO], out[M.GEMM_IMAD]))
