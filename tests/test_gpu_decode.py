"""hann_decrypt_scores / hann_decrypt_compact on ciphertexts that are plaintexts (c1 = 0) of chosen integers: the CRT has to give every
centred integer exactly, rounded to binary64 once, for every chain length and for integers at the ends of their range.  Constant
polynomials show that bit for bit; the slots of full ones are compared with a binary64 FFT of the exactly rounded coefficients."""
import random

import numpy as np
import pytest

from oracle.oracle import find_primes
from paper_2608_21131_b200 import synth

pytestmark = pytest.mark.gpu


def slots(coeffs, logN):
    """sum over k of m_k zeta_j^k at the canonical slots, from n complex numbers (m_k + i m_{k+n}) exp(i pi k / N)"""
    n, N = 1 << (logN - 1), 1 << logN
    a = (coeffs[:n] + 1j * coeffs[n:]) * np.exp(1j * np.pi * np.arange(n) / N)
    u, g = [], 1
    for _ in range(n):
        u.append((g - 1) // 4)
        g = g * 5 % (2 * N)
    return (n * np.fft.ifft(a))[u]


@pytest.mark.parametrize("logN,bits,count", [(4, (50,), 1), (5, (62, 61), 3), (9, (50, 45, 40), 9), (10, (50,) * 4, 17), (9, (58, 45, 45, 45, 45), 2),
                                             (11, (45,) * 9, 2), (10, (61,) * 15, 1)])
def test_decoded_slots_of_chosen_integers(logN, bits, count):
    from paper_2608_21131_b200 import binding as b

    q = []
    for w in bits:
        q.append(next(x for x in find_primes(w, logN + 1, 16) if x not in q))
    p = next(x for x in find_primes(60, logN + 1, 16) if x not in q)
    ps = synth.ParamSet("dec", logN, tuple(q), p, 20, 4, 2, 0)
    c = b.Context(ps)
    N, L = ps.N, ps.L
    s = synth.key_material(ps, 1, rots=[]).s
    rng = random.Random(logN * 100 + L)
    for limbs, rescaled in [(L, False)] + ([(max(1, L - 1), True)] if L > 1 else []):
        Q = 1
        for x in q[:limbs]:
            Q *= x
        ct = np.zeros((count, 2, limbs, N), dtype=np.uint64)
        mult, log_scale = (q[-1] if rescaled else 1), Q.bit_length()
        exact = np.zeros((count, N))
        for i in range(count):
            # the ends of the range, small integers, numbers halfway between two binary64, then uniform ones of every size
            m = [Q // 2, -(Q // 2), 0, 1, -1, (1 << 53) + 1, -(1 << 53) - 1, 3 << 52]
            m += [rng.randrange(-(Q // 2), Q // 2 + 1) >> rng.randrange(0, Q.bit_length()) for _ in range(N - len(m))]
            m = [(x + Q // 2) % Q - Q // 2 for x in m]
            for l in range(limbs):
                ct[i, 0, l] = [x % q[l] for x in m]
            exact[i] = [x * mult / (1 << log_scale) for x in m]  # a quotient of integers is rounded once
        if rescaled:
            got, imag = c.decrypt_compact(s, ct, True, log_scale_in=log_scale, want_imag=True)
        else:
            got, imag = c.decrypt_scores(s, ct, log_scale_out=log_scale, want_imag=True)
        for i in range(count):
            want = slots(exact[i], logN)
            # logN - 1 butterfly stages and the twist, each a rounding or two of relative size 2^-53, on either side
            assert np.linalg.norm(got[i] + 1j * imag[i] - want) <= 8 * logN * 2.0 ** -53 * np.linalg.norm(want)


def test_scratch_of_a_decryption_is_bounded():
    """eight ciphertexts of fifteen primes at N = 2^16 go through in pieces: the context's device memory grows by no more than the 64 MiB
    that the header gives, and every ciphertext decrypts to the bits it has on its own"""
    import torch

    from paper_2608_21131_b200 import binding as b

    q = find_primes(45, 17, 15)
    ps = synth.ParamSet("deep", 16, tuple(q), find_primes(60, 17, 1)[0], 20, 4, 2, 0)
    c = b.Context(ps)
    s = synth.key_material(ps, 1, rots=[]).s
    ct = np.random.default_rng(5).integers(0, min(q), size=(8, 2, ps.L, ps.N), dtype=np.uint64)
    alone = [c.decrypt_scores(s, ct[i:i + 1], log_scale_out=640, want_imag=True) for i in range(8)]
    free = torch.cuda.mem_get_info()[0]
    got, imag = c.decrypt_scores(s, ct, log_scale_out=640, want_imag=True)
    assert free - torch.cuda.mem_get_info()[0] <= 64 << 20
    for i in range(8):
        assert np.array_equal(got[i], alone[i][0][0]) and np.array_equal(imag[i], alone[i][1][0])


def chain_context(logN, bits):
    from paper_2608_21131_b200 import binding as b

    q = []
    for w in bits:
        q.append(next(x for x in find_primes(w, logN + 1, 16) if x not in q))
    p = next(x for x in find_primes(60, logN + 1, 16) if x not in q)
    ps = synth.ParamSet("dec", logN, tuple(q), p, 20, 4, 2, 0)
    return b.Context(ps), q, synth.key_material(ps, 1, rots=[]).s


def decode(c, s, q, limbs, polys, log_scale):
    """real and imaginary slots of plaintext polynomials (lists of integers) over the first `limbs` primes"""
    ct = np.zeros((len(polys), 2, limbs, c.N), dtype=np.uint64)
    for i, m in enumerate(polys):
        for l in range(limbs):
            ct[i, 0, l, : len(m)] = [x % q[l] for x in m]
    if limbs < len(q):
        return c.decrypt_compact(s, ct, True, log_scale_in=log_scale, want_imag=True)
    return c.decrypt_scores(s, ct, log_scale_out=log_scale, want_imag=True)


CHAINS = [(50,), (62, 61), (50, 45, 40), (58, 45, 45, 45), (45,) * 5, (61,) * 8, (50,) * 9, (61,) * 15]


@pytest.mark.parametrize("bits", CHAINS)
def test_a_constant_decodes_to_the_nearest_binary64(bits):
    """the constant polynomial m has m in every slot: the twiddle of the first coefficient is 1 and every other term of the transform is a
    zero, so the real parts are the rounded integer itself, bit for bit, with nothing of its size beside it to hide an error"""
    c, q, s = chain_context(4, bits)
    for limbs in {len(q), max(1, len(q) - 1)}:
        Q = 1
        for x in q[:limbs]:
            Q *= x
        m = [1, 2, 3, (1 << 53) - 1, 1 << 53, (1 << 53) + 1, (1 << 53) + 3, Q // 2, Q // 2 - 1, Q // 3]
        for k in range(1, Q.bit_length() - 56):
            # halfway to the even and to the odd neighbour, and one unit (in the lowest word) to either side
            for tie in ((1 << 53) + 1, (1 << 53) + 3, (1 << 54) - 1):
                m += [tie << k, (tie << k) + 1, (tie << k) - 1]
        m = [x for x in m if x <= Q // 2]
        m += [-x for x in m] + [0]
        mult, log_scale = (q[-1] if limbs < len(q) else 1), 30
        got, imag = decode(c, s, q, limbs, [[x] for x in m], log_scale)
        for i, x in enumerate(m):
            want = x * mult / (1 << log_scale)  # a quotient of integers is rounded once, to nearest even
            assert np.all(got[i] == want) and np.all(imag[i] == 0), (limbs, i, x)


@pytest.mark.parametrize("bits", CHAINS)
def test_small_integers_under_a_long_chain(bits):
    """coefficients of twenty bits, far below the chain's product: the error is relative to them"""
    c, q, s = chain_context(9, bits)
    rng = random.Random(len(bits))
    m = [[rng.randrange(-(1 << 20), (1 << 20) + 1) for _ in range(c.N)] for _ in range(3)]
    got, imag = decode(c, s, q, len(q), m, 10)
    for i in range(3):
        want = slots(np.array(m[i], dtype=np.float64) / 1024, 9)
        # as in test_decoded_slots_of_chosen_integers
        assert np.linalg.norm(got[i] + 1j * imag[i] - want) <= 8 * 9 * 2.0 ** -53 * np.linalg.norm(want)
