"""Operands that show a shift-group sum kept too long in fp32, and the check on
the host that they do.

All digits are -128 (each product +2^14) except that row i of A holds the digits
(1, 1, 1, 1) at one place of stage i mod S and row j of B the digits (1, 0, 0, 0)
at the same place of stage j mod S (a stage is 32 K).  Where the two meet (i = j
mod S) every shift group gains exactly one odd product, and everything else it
sums is a multiple of 128: it stays exact up to 2^24 and rounds above.  So one
stage beyond the 8 that groups 2 and 3 may gather, or the 16 of groups 0 and 1,
is lost, wherever the odd term lies in it."""
import numpy as np
import pytest

STAGE = 32
PLACE = 3                      # of a stage, so that a last stage of 5 K holds it too
ALL_M128 = 0x7F7F7F80          # digits (-128, -128, -128, -128)
ONES = 0x01010101              # digits (1, 1, 1, 1)
ONE = 0x00000001               # digits (1, 0, 0, 0)


def drain_operands(rows_a, rows_b, K):
    """(A, B, S): row i of A depends on i mod S only, row j of B on j mod S."""
    S = (K + STAGE - 1) // STAGE
    A = np.full((rows_a, K), ALL_M128, np.uint32)
    B = np.full((rows_b, K), ALL_M128, np.uint32)
    i, j = np.arange(rows_a), np.arange(rows_b)
    A[i, STAGE * (i % S) + PLACE] = ONES
    B[j, STAGE * (j % S) + PLACE] = ONE
    return A, B, S


def digits(x):
    b = (x.astype(np.uint64) + 0x80808080) & 0xFFFFFFFF
    return [((b >> np.uint64(8 * d)) & np.uint64(0xFF)).astype(np.int64) - 128 for d in range(4)]


def group_sum(a, b, s):
    """Shift group s of one output: (exact sum, sum in fp32 in steps of 16 K)."""
    da, db = digits(a), digits(b)
    p = sum(da[i] * db[s - i] for i in range(s + 1)).reshape(-1, 16).sum(1)
    acc = np.float32(0)
    for v in p:
        acc = np.float32(acc + np.float32(v))
    return int(p.sum()), int(acc)


@pytest.mark.parametrize("pair,limit", [((0, 1), 16), ((2, 3), 8)])
def test_a_window_beyond_the_limit_rounds(pair, limit):
    for stages in (limit, limit + 1):
        A, B, S = drain_operands(stages, stages, STAGE * stages)
        exact = [all(x == y for x, y in (group_sum(A[i], B[i], s) for s in pair)) for i in range(S)]
        assert all(exact) if stages == limit else not any(exact), (stages, exact)
        assert all(x == y for x, y in (group_sum(A[0], B[1], s) for s in pair))   # no odd term: never seen
