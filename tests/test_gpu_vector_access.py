"""Kernels that move two or four words a thread: the automorphism's pairs for
every kind of Galois element (in order and swapped), the smallest ring, and
stage buffers that are only 8-byte aligned, against the oracle."""
import numpy as np
import pytest

from oracle import oracle as orc
from paper_2311_01598_gb300 import inputs
from tests._gpu import built_lib, need_gpu, pair

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("logN", [10, 13])
@pytest.mark.parametrize("offset", [0, 1])
def test_automorph(logN, offset):
    torch = need_gpu()
    ks = built_lib()
    P, C = pair(logN, 3, 1, 3)
    N = C.N
    a = inputs.uniform_towers(C.q, N, seed=5)
    buf = torch.zeros(3 * N + 2, dtype=torch.int64, device="cuda")
    src = buf[offset:offset + 3 * N].view(3, N)
    src.copy_(ks.to_device(a))
    for g in (1, 3, 5, N - 1, N + 1, 2 * N - 1, pow(5, 77, 2 * N)):
        want = np.stack([orc.automorph_eval(a[t], logN, g) for t in range(3)])
        outb = torch.zeros(3 * N + 2, dtype=torch.int64, device="cuda")
        out = outb[offset:offset + 3 * N].view(3, N)
        P.automorph(0, g, src, out)
        assert np.array_equal(ks.to_host(out), want), g
        P.automorph(0, g, src, out, accumulate=True)
        q = np.array(C.q, dtype=np.uint64)[:, None]
        assert np.array_equal(ks.to_host(out), (want + want) % q), g
        assert int(outb[3 * N + offset]) == 0


@pytest.mark.parametrize("offset", [0, 1])
def test_moddown_output(offset):
    torch = need_gpu()
    ks = built_lib()
    P, C = pair(10, 5, 2, 2)
    cp = inputs.uniform_towers(C.q[:4] + C.p, C.N, seed=9)
    outb = torch.zeros(4 * C.N + 2, dtype=torch.int64, device="cuda")
    out = outb[offset:offset + 4 * C.N].view(4, C.N)
    P.moddown(4, ks.to_device(cp), out)
    assert np.array_equal(ks.to_host(out), C.moddown(4, cp))


@pytest.mark.parametrize("compressed", [False, True])
def test_hoisted_levels(compressed):
    need_gpu()
    ks = built_lib()
    P, C = pair(10, 7, 3, 3)
    s = inputs.ternary_secret(C.N, 3)
    gals = [1, 3, 2 * C.N - 1] + inputs.galois_elements(C.N, 2, 4)
    gen = P.keygen_compressed if compressed else P.keygen
    ref = C.keygen_compressed if compressed else C.keygen
    keys = [gen(s, inputs.galois_secret(s, g), seed=50 + i) for i, g in enumerate(gals)]
    evks = [ref(s, inputs.galois_secret(s, g), seed=50 + i) for i, g in enumerate(gals)]
    for nact in (1, 4, 7):
        d = inputs.uniform_towers(C.q[:nact], C.N, seed=60 + nact)
        o0 = [ks.empty((nact, C.N)) for _ in gals]
        o1 = [ks.empty((nact, C.N)) for _ in gals]
        P.switch_hoisted(keys, gals, nact, ks.to_device(d), o0, o1)
        for w0, w1, a, b in zip(*C.keyswitch_hoisted(nact, d, evks, gals), o0, o1):
            assert np.array_equal(ks.to_host(a), w0) and np.array_equal(ks.to_host(b), w1)
