"""The NTT butterfly forms a parameter set's primes select: sets just below a
power of two (the default prime rule) take the quotient-free product, others
the general one.  The product's bounds on the CPU with Python integers, and
GPU transforms against the oracle at the edges of the forms: smallest and
largest bit lengths, the sets whose transforms fold at each place, the largest
prime gap of a set (its last tower) and extreme residues."""
import random

import numpy as np
import pytest

from oracle import oracle as orc
from tests._gpu import built_lib, need_gpu


def _mul(a, w, q, b):
    """The kernels' product, word by word, with every intermediate checked to fit its register."""
    k, M32, M64 = b - 31, (1 << 32) - 1, (1 << 64) - 1
    c2 = (1 << (b + 1)) - 2 * q
    w2 = (w << 32) % q
    wl, wh, vl, vh = w & ((1 << k) - 1), w >> k, w2 & ((1 << k) - 1), w2 >> k
    a0, a1 = a & M32, a >> 32
    m1 = a0 * wh + a1 * vh
    m0 = a0 * wl + a1 * vl
    assert max(wh, vh) < 1 << 31 and c2 <= M32 and m1 <= M64 and m0 <= M64
    t = m0 + ((m1 & M32) << k) + (m1 >> 32) * c2
    assert t <= M64
    return t, c2


@pytest.mark.parametrize("logN,bits,towers", [(10, 40, 6), (12, 50, 4), (16, 54, 32), (17, 54, 60), (17, 56, 96)])
def test_product_bounds(logN, bits, towers):
    primes = orc.gen_primes(logN, bits, towers)
    r = random.Random(logN)
    edge = [0, 1, (1 << 32) - 1, 1 << 32, (1 << 63), (1 << 64) - 1]
    for q in (primes[0], primes[-1]):
        for w in [0, 1, q - 1, q // 2] + [r.randrange(q) for _ in range(50)]:
            for a in edge + [r.randrange(1 << 64) for _ in range(50)]:
                t, c2 = _mul(a, w, q, bits)
                assert t % q == a * w % q
                assert t <= ((1 << 32) - 1) * c2 + 6 * (1 << bits)


@pytest.mark.gpu
@pytest.mark.parametrize("cluster", [0, 1])
@pytest.mark.parametrize("logN,bits,nq,kp", [(10, 30, 3, 1), (10, 40, 3, 1), (12, 50, 3, 1), (13, 56, 6, 2),
                                             (16, 54, 24, 8), (16, 56, 50, 10), (17, 50, 45, 15), (17, 54, 45, 15),
                                             (17, 56, 64, 32)])
def test_transforms(logN, bits, nq, kp, cluster):
    need_gpu()
    ks = built_lib()
    P = ks.Params(logN, nq, kp, min(nq, 3), prime_bits=bits)
    P.set_ntt_cluster(cluster)
    primes = P.q + P.p
    N = 1 << logN
    rng = np.random.Generator(np.random.PCG64(7 * logN + bits))
    for t in (0, nq - 1, nq, nq + kp - 1):
        q = primes[t]
        psi = orc.find_psi(q, logN)
        ones = np.full(N, q - 1, dtype=np.uint64)
        alt = ones.copy()
        alt[::2] = 0
        half = ones.copy()
        half[: N // 2] = 0
        for a in (ones, alt, half, rng.integers(0, q, size=N, dtype=np.uint64)):
            x = ks.to_device(a[None, :])
            P.ntt(t, x, inverse=False)
            assert np.array_equal(ks.to_host(x)[0], orc.ntt(a, logN, q, psi)), f"forward, tower {t}"
            x = ks.to_device(a[None, :])
            P.ntt(t, x, inverse=True)
            assert np.array_equal(ks.to_host(x)[0], orc.intt(a, logN, q, psi)), f"inverse, tower {t}"
