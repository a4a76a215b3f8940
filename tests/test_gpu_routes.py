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
