"""The index folding of the compile-time fixed-point lines (passes_fixed.cuh, FixedLine), checked on the
CPU for every length, stage, thread and butterfly: shared-memory addresses formed as a per-thread base
plus a compile-time offset equal the padded addresses e + (e >> 3) of the plain Stockham indices,
each stage's outputs cover the line once, no address passes the padded line, and every twiddle entry a
stage reads lies on the side (shared-memory copy or whole table) it is read from, with the power it
stands for.
"""
import numpy as np
import pytest

LENGTHS = [512, 1024, 2048, 4096, 8192]


def pidx(e):
    return e + (e >> 3)


def padded(L):
    return L + (L >> 3) + 1


def radices(L):
    l2 = L.bit_length() - 1
    return [16] * (l2 // 4) + ([1 << (l2 % 4)] if l2 % 4 else [])


def variants(R):
    return 3 if R == 16 else (2 if R in (8, 5) else 1)


def table(L):
    """Offsets of the stages' blocks, and for each entry the exponent e of exp(-2 pi i e / L)."""
    toff, power, Ns = [], [], 1
    for s, R in enumerate(radices(L)):
        toff.append(len(power))
        if s:
            for _ in range(variants(R)):
                for q in range(1, R):
                    power += [q * k * (L // (Ns * R)) % L for k in range(L // 4 if (L, R) == (8192, 2) else Ns)]
        Ns *= R
    return toff, power


def shared_entries(L):
    return 720 + {512: 256, 1024: 768, 2048: 3584, 4096: 3840, 8192: 3840}[L]


@pytest.mark.parametrize("L", LENGTHS)
def test_addresses_match_the_stockham_indices(L):
    TPT, R = L // 16, radices(L)
    lt = np.arange(TPT)

    def at(c):  # FixedLine::at
        assert c % 8 == 0
        return pidx(lt) + c + (c >> 3)

    for q in range(16):
        assert np.array_equal(at(q * TPT), pidx(lt + q * TPT))
    for p in range(16):  # store0
        assert np.array_equal(18 * lt + p + (p >> 3), pidx(16 * lt + p))
    Ns = 16
    for s in range(1, len(R) - 1):  # mids
        assert R[s] == 16 and Ns == 1 << (4 * s)
        k = lt & (Ns - 1)
        o, st = ((lt >> (4 * s)) << (4 * s + 4)) + k, Ns + (Ns >> 3)
        outs = []
        for p in range(16):
            direct = (lt // Ns) * 16 * Ns + lt % Ns + p * Ns
            assert np.array_equal(pidx(o) + p * st, pidx(direct))
            outs.append(direct)
        assert np.array_equal(np.sort(np.concatenate(outs)), np.arange(L))
        Ns *= 16
    r = R[-1]
    NB = 16 // r
    assert Ns == L // r  # last
    outs = []
    for b in range(NB):
        j = lt + b * TPT
        assert j.max() < Ns
        for q in range(r):
            assert np.array_equal(at(b * TPT + q * Ns), pidx(j + q * Ns))
            outs.append(j + q * Ns)
    assert np.array_equal(np.sort(np.concatenate(outs)), np.arange(L))
    assert pidx(L - 1) < padded(L)


@pytest.mark.parametrize("L", LENGTHS)
def test_twiddles_are_read_from_where_they_lie(L):
    TPT, R = L // 16, radices(L)
    toff, power = table(L)
    smem, whole = shared_entries(L), L <= 2048
    assert len(power) == smem if whole else len(power) > smem
    Ns = 16
    for s in range(1, len(R)):
        r = R[s]
        last = s == len(R) - 1
        NB = 16 // r if last else 1
        for copy in range(variants(r)):
            for b in range(NB):
                j = np.arange(TPT) + b * TPT
                k = j if last else j & (Ns - 1)
                turn = 0
                if L == 8192 and last and b >= NB // 2:  # w^(k + L/4) = -i w^k
                    k, turn = j - L // 4, L // 4
                o = toff[s] + copy * (r - 1) * Ns + k
                for q in range(1, r):
                    i = o + (q - 1) * Ns
                    assert i.min() >= 0 and i.max() < len(power)
                    assert np.array_equal((np.array(power)[i] + turn) % L, q * (j if last else k) * (L // (Ns * r)) % L)
                    if not whole:  # one pointer serves all of a butterfly's entries
                        assert np.array_equal(i < smem, o < smem)
        Ns *= r
