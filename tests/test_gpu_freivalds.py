"""Freivalds integrity check (Sec. 3.2 box, Init W step 4 and Online step 4;
appendix "Computational integrity") through the C ABI against the oracle:
the check vectors and a^T W' bit-exact, honest answers accepted, a corrupted
entry of Y' flagged on exactly its token."""
import numpy as np
import pytest

import oracle as O
from paper_2607_29221_gb300 import workloads as wl

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

KEY = wl.mask_key()


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2607_29221_gb300 import build
    build.build()
    yield


def _host(t):
    torch.cuda.synchronize()
    return t.cpu().numpy().view(np.uint32)


@pytest.mark.parametrize("m,n,l,k", [(128, 256, 64, 4), (131, 300, 9, 3), (200, 256, 1, 16),
                                     (1000, 512, 300, 8)])
def test_freivalds_matches_oracle_and_detects(m, n, l, k):
    from paper_2607_29221_gb300 import mosaic as M
    from paper_2607_29221_gb300 import protocol as PR
    op = O.Params(d=3, r=(96, 64, 40), t=(8, 4))
    gp = M.default_params(d=3, r=[96, 64, 40], t=[0, 8, 4])
    proto = PR.Protocol(KEY, gp, variant=M.GEMM_AUTO)
    W = wl.weights(m, n, std=1.0)
    X = wl.activations(l, n)
    ch = PR.Chains(proto, PR.pad_width(n))
    layer = PR.SecureLinear(proto, torch.from_numpy(W).cuda(), 7, ch)
    layer.freivalds_setup(k)
    mp = layer.init_x(l, 11)
    Xp, s_x, Xpl = layer.mask_input(torch.from_numpy(X).cuda(), mp)
    Z = layer.server(Xp, Xpl)
    ref = O.secure_linear(KEY, op, W, X.T.copy(), matrix_id=7, pass_id=11)
    a, Yc = O.freivalds_setup(KEY, op, ref["ws"], 7, k)
    assert np.array_equal(_host(layer.check_a), a)
    assert np.array_equal(_host(layer.check_Y), Yc)
    bad, n_bad = layer.freivalds_check(Z, Xp)
    M.mosaic_device_status()
    assert _host(n_bad)[0] == 0 and not np.any(_host(bad))
    # an odd error in Y'[j][i] is caught by every vector (a_v[i] != 0)
    j, i = l // 2, m // 3
    Zc = Z.clone()
    Zc[j, i] += 977
    bad, n_bad = layer.freivalds_check(Zc, Xp)
    got = _host(bad)
    want = O.freivalds_check(a, Yc, _host(Zc)[:, :m].T.copy(), ref["X_masked"])
    assert np.array_equal(got, want)
    assert got[j] == np.count_nonzero(a[:, i]) and np.count_nonzero(got) == 1
    assert _host(n_bad)[0] == 1
    # the Q columns of Z are not covered by the check
    if l > 1:
        Zq = Z.clone()
        Zq[0, m] += 1
        bad, n_bad = layer.freivalds_check(Zq, Xp)
        assert _host(n_bad)[0] == 0


# Both token groupings (below and from 76 tokens), every cluster split, ragged
# groups, all vector-count steps, columns fewer than a share, and strides that
# forbid 16-byte loads of one or both operands.
@pytest.mark.parametrize("l,m,n,k,dz,dx", [
    (1, 17, 4, 16, 0, 0), (1, 4096, 8192, 1, 0, 0), (5, 100, 64, 2, 3, 0), (75, 333, 257, 3, 1, 1),
    (76, 64, 32, 4, 0, 4), (77, 1000, 96, 5, 5, 0), (303, 130, 131, 8, 2, 2), (610, 40, 64, 9, 0, 0),
    (1300, 52, 36, 16, 4, 0)])
def test_check_counts_differing_vectors(l, m, n, k, dz, dx):
    from paper_2607_29221_gb300 import mosaic as M
    rng = np.random.default_rng(l * 31 + k)
    u32 = lambda *s: rng.integers(0, 1 << 32, s, dtype=np.uint32)
    a, Yc, Z, X = u32(k, m), u32(k, n), u32(l, m + dz), u32(l, n + dx)
    a[:, :k] = np.eye(k, dtype=np.uint32)
    # Honest answers: column v < k is chosen so that vector v agrees; then a third of the tokens is tampered with.
    Z[:, :k] = X[:, :n] @ Yc.T - Z[:, k:m] @ a[:, k:].T
    off = rng.integers(0, l, l // 3 + 1)
    Z[off, rng.integers(0, m, len(off))] += np.uint32(1 << 31)
    want = np.count_nonzero(Z[:, :m] @ a.T != X[:, :n] @ Yc.T, axis=1)
    dev = lambda x: torch.from_numpy(x.view(np.int32)).cuda()
    bad = torch.full((l,), -1, dtype=torch.int32, device="cuda")
    n_bad = torch.full((1,), 7, dtype=torch.int32, device="cuda")
    ws = torch.empty(M.mosaic_workspace_bytes(M.OP_FREIVALDS_CHECK, k, 0, l), dtype=torch.uint8, device="cuda")
    M.mosaic_freivalds_check(k, dev(a), dev(Yc), m, n, l, dev(Z), m + dz, dev(X), n + dx, bad, n_bad, ws)
    assert np.array_equal(_host(bad), want.astype(np.uint32))
    assert _host(n_bad)[0] == 7 + np.count_nonzero(want)
