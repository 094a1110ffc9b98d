"""The warp-per-line kernel's choice of shared-memory swizzle against a count of
bank conflicts in the walk its lanes take (host code, no GPU)."""
import ctypes

import pytest

import paper_1008_0861_gb300 as P
from paper_1008_0861_gb300 import build


def _wavefronts(N, n, team, code):
    """Sum over steps and quarter warps of the most lanes on one bank group: lane
    t goes down its segment from the last chunk."""
    m = -(-n // N)
    U, rr = divmod(m, team)
    log_u = U.bit_length() - 1
    shift, mask = (code - 1 if code >= 2 else log_u), (0 if code == 1 else 7)
    total = 0
    for k in range(U + (rr > 0)):
        for q in range(0, team, 8):
            count = [0] * 8
            for t in range(q, q + 8):
                length = U + (t < rr)
                if k < length:
                    c = t * U + min(t, rr) + length - 1 - k
                    count[(c ^ ((c >> shift) & mask) if c < (m & ~7) else c) & 7] += 1
            total += max(count)
    return total


@pytest.mark.parametrize("prec,n,team", [(1, 196, 8), (1, 228, 8), (1, 256, 16), (1, 348, 16), (1, 512, 32), (1, 916, 32),
                                         (1, 1001, 32), (1, 2008, 32), (0, 98, 8), (0, 176, 16), (0, 606, 32), (0, 1024, 32)])
def test_the_choice_has_the_fewest_wavefronts(prec, n, team):
    build.build()
    choose = P.load()._ZN5aniso13line4_swizzleEiii
    code = choose(prec, n, team)
    N = 2 if prec == 0 else 4
    assert _wavefronts(N, n, team, code) == min(_wavefronts(N, n, team, c) for c in range(8))
