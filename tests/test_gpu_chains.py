"""Public chains on the GPU with the full workspace (tensor-core products from
digit planes of the second factor's transpose) and with the minimum one
(CUDA-core products): both bit-identical to the oracle's chains."""
import numpy as np
import pytest

import oracle as O
from paper_2607_29221_gb300 import workloads as wl

pytestmark = pytest.mark.gpu
KEY = wl.mask_key()


def _up(v):
    return (v + 255) // 256 * 256


# Widths of one and several 32-column blocks; ranks that are no multiple of 8, 32 or 64 (ragged
# digit quads and K tails), tiny ones, and the Example 3.1 ranks.
@pytest.mark.parametrize("n_pad,r,t", [
    (32, (5, 3, 2), (0, 1, 1)), (64, (70, 33, 9), (0, 4, 4)), (128, (64, 63, 65), (0, 4, 4)),
    (512, (1536, 1024, 652), (0, 80, 80)), (256, (300, 129), (0, 4)), (128, (40,), (0,))])
def test_chains_match_oracle_for_both_workspaces(n_pad, r, t):
    import torch

    from paper_2607_29221_gb300 import mosaic as M
    d = len(r)
    p = M.default_params(d=d, r=r, t=t)
    po = O.Params(d=d, r=r, t=t[1:])
    key = M.make_key(KEY)
    Sr = sum(r)
    Po, Co = O.chains(KEY, po, n_pad)
    full = M.mosaic_workspace_bytes(M.OP_MASK_CHAINS, 0, n_pad, 0, p)
    minimum = sum(2 * _up(4 * r[i] * r[i - 1]) for i in range(1, d))
    assert full >= minimum
    for size in {full, minimum}:
        P, C, CT = (torch.zeros(s, dtype=torch.int32, device="cuda") for s in ((Sr, n_pad), (n_pad, Sr), (Sr, n_pad)))
        ws = torch.empty(max(size, 1), dtype=torch.uint8, device="cuda")
        M.mosaic_mask_chains(p, key, n_pad, n_pad, P, C, CT, ws[:size] if size else ws)
        M.mosaic_device_status()
        P, C, CT = (x.cpu().numpy().view(np.uint32) for x in (P, C, CT))
        assert np.array_equal(P, np.vstack(Po)), size
        assert np.array_equal(C, np.hstack(Co)), size
        assert np.array_equal(CT, C.T), size
