"""Index proof of the run-time-length path's slot layout and last pass (kd_generic.cuh), on the
host, for every supported length: the padded addresses are distinct, a group of any pass is an
arithmetic progression from its base, and the items of the last pass cover every frequency
once with the lower one of each pair first, within the 2 R bits of their sign mask."""

import pytest

RADICES = (16, 8, 4, 2, 9, 3, 5, 7, 11, 13, 43)


def _plan(n):
    R, rem = [], n
    for r in RADICES:
        while rem % r == 0:
            R.append(r)
            rem //= r
    if rem != 1:
        return None
    S, b = [], n
    for r in R:
        b //= r
        S.append(b)
    P, size = [0] * len(R), 1
    for i in reversed(range(len(R))):
        P[i] = 1 if i == len(R) - 1 else size | 1
        size = P[i] * R[i]
    return R, S, P, size


def _address(s, S, P):
    at = 0
    for si, pi in zip(S, P):
        at += s // si * pi
        s %= si
    return at


@pytest.mark.parametrize("lo,hi", [(1, 700), (700, 2100), (5120, 5121), (13824, 13825), (16380, 16385)])
def test_addresses_and_groups(lo, hi):
    for n in range(lo, hi):
        plan = _plan(n)
        if plan is None:
            continue
        R, S, P, size = plan
        addr = [_address(s, S, P) for s in range(n)]
        assert len(set(addr)) == n and (n == 1 or max(addr) < size <= 65535)
        B = n
        for r, s, p in zip(R, S, P):
            for g in range(n // r):
                base = g // s * B + g % s
                assert all(addr[base + j * s] == addr[base] + j * p for j in range(r))
            B = s


def test_last_pass_covers_every_frequency():
    for n in range(2, 3000):
        plan = _plan(n)
        if plan is None or plan[0][-1] > 16:
            continue
        R = plan[0][-1]
        M, h = n // R, (R + 1) // 2
        seen = []
        for p in range(M // 2 + 1):
            if 0 < p and 2 * p < M:
                pairs = [(p + M * j, M - p + M * (R - 1 - j)) for j in range(h)]
                pairs += [(M - p + M * j, p + M * (R - 1 - j)) for j in range(R // 2)]
                bits = list(range(h)) + [h + j for j in range(R // 2)]
            elif p == 0:
                pairs = [(0, 0)] + [(M * j, M * (R - j)) for j in range(1, h)]
                bits = list(range(h))
                if R % 2 == 0:
                    pairs.append((M * R // 2, M * R // 2))
                    bits.append(R // 2)
            else:
                pairs = [(p + M * j, p + M * (R - 1 - j)) for j in range(R // 2)]
                bits = list(range(R // 2))
                if R % 2 == 1:
                    pairs.append((p + M * (R // 2), p + M * (R // 2)))
                    bits.append(R // 2)
            assert len(set(bits)) == len(bits) and max(bits) < R
            for (k, m), q in zip(pairs, bits):
                assert (k + m) % n == 0 and (2 * k < n or (k == m and 2 * k in (0, n)))
                # the frequency that the staged mask holds at this bit
                if not (p == 0 and R % 2 == 0 and q == R // 2):
                    assert k == (p + M * q if q < h else M - p + M * (q - h))
                seen += [k] if k == m else [k, m]
        assert sorted(seen) == list(range(n))
