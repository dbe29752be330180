"""The index proof of tests/test_generic_tables.py for every supported length up to 16384 (there:
addresses below 2100 and a few more, the last pass below 3000), with arrays."""

import numpy as np
import pytest

from tests.test_generic_tables import _plan

LENGTHS = [n for n in range(1, 16385) if _plan(n) is not None]


def _addresses(s, S, P):
    at = np.zeros_like(s)
    for si, pi in zip(S, P):
        at += s // si * pi
        s = s % si
    return at


@pytest.mark.parametrize("part", range(8))
def test_addresses_and_groups(part):
    assert len(LENGTHS) > 1000
    for n in LENGTHS[part::8]:
        R, S, P, size = _plan(n)
        addr = _addresses(np.arange(n), S, P)
        assert np.unique(addr).size == n and (n == 1 or addr.max() < size <= 65535)
        B = n
        for r, s, p in zip(R, S, P):
            g = np.arange(n // r)
            base = g // s * B + g % s
            for j in range(1, r):
                assert (addr[base + j * s] == addr[base] + j * p).all()
            B = s


@pytest.mark.parametrize("part", range(8))
def test_last_pass_covers_every_frequency(part):
    for n in LENGTHS[part::8]:
        R = _plan(n)[0][-1] if n > 1 else 0
        if n < 2 or R > 16:
            continue
        M, h = n // R, (R + 1) // 2
        p = np.arange(M // 2 + 1)
        seen = np.zeros(n, dtype=int)

        def pairs(k, m, bit):
            """Pairs (k, n - k) at mask bit `bit`, the lower frequency first."""
            assert ((k + m) % n == 0).all() and ((2 * k < n) | ((k == m) & (2 * k == n)) | (k == 0)).all()
            assert 0 <= bit < R
            np.add.at(seen, k, 1)
            np.add.at(seen, m[m != k], 1)

        mid = p[(p > 0) & (2 * p < M)]
        for j in range(h):
            pairs(mid + M * j, M - mid + M * (R - 1 - j), j)
        for j in range(R // 2):
            pairs(M - mid + M * j, mid + M * (R - 1 - j), h + j)
        zero = np.zeros(1, dtype=int)
        pairs(zero, zero, 0)
        for j in range(1, h):
            pairs(zero + M * j, zero + M * (R - j), j)
        if R % 2 == 0:
            pairs(zero + M * R // 2, zero + M * R // 2, R // 2)
        if M % 2 == 0:
            c = zero + M // 2
            for j in range(R // 2):
                pairs(c + M * j, c + M * (R - 1 - j), j)
            if R % 2 == 1:
                pairs(c + M * (R // 2), c + M * (R // 2), R // 2)
        assert (seen == 1).all()
