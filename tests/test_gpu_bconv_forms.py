"""Which forms a parameter set's primes select: the tensor-core base conversion's
Montgomery epilogue at its source limits (sets that are not just below a power
of two: primes k*2^32 + 1, 40-bit default sets), the folding epilogue at the
smallest bit lengths that allow it, lists of two bit lengths (quotient-free
butterflies, Montgomery epilogue) and lists that one prime keeps from the
quotient-free form.  The tensor cores are asked for, so that a set's size does
not choose the engine; largest operands and uniform ones, against the oracle."""
import numpy as np
import pytest

from oracle import oracle as orc
from paper_2311_01598_gb300 import inputs
from tests._gpu import built_lib, need_gpu
from tests.test_gpu_edges import max_evk, max_w_cprime, max_y_input, random_evk

pytestmark = pytest.mark.gpu


def _below(logN, top, n):
    """The n largest primes = 1 mod 2N below top."""
    out, x = [], top - (top - 1) % (2 << logN)
    while len(out) < n:
        if x < top and all(pow(a, x - 1, x) == 1 for a in (2, 3, 5, 7, 11, 13, 17)):
            out.append(x)
        x -= 2 << logN
    return out


def _list(form, logN, n):
    if form.startswith("special"):
        return built_lib().special_primes(int(form[7:]), n)
    if form.startswith("mixed"):  # two bit lengths, both just below a power of two
        a, b = map(int, form[5:].split("_"))
        return [x for two in zip(_below(logN, 1 << a, n), _below(logN, 1 << b, n)) for x in two][:n]
    if form == "off54":  # one prime three quarters up
        return _below(logN, 1 << 54, n - 1) + _below(logN, 3 << 52, 1)
    if form == "above54":  # just above the power of two
        return _below(logN, (1 << 53) + (1 << 30), n)
    return _below(logN, 1 << int(form), n)


@pytest.mark.parametrize("form,logN,nq,kp,dnum", [
    ("special54", 11, 9, 9, 1), ("special54", 12, 10, 10, 1), ("special54", 11, 18, 18, 1), ("special56", 11, 9, 9, 1),
    ("special56", 12, 18, 18, 1), ("special56", 11, 19, 19, 1), ("special56", 13, 24, 8, 3),
    ("40", 11, 8, 3, 2), ("40", 12, 9, 9, 1), ("40", 10, 18, 18, 1), ("42", 10, 8, 3, 2), ("44", 10, 10, 10, 1),
    ("47", 12, 19, 19, 1), ("mixed54_50", 12, 9, 9, 1), ("mixed56_54", 11, 18, 10, 1), ("mixed55_52", 16, 8, 3, 2),
    ("off54", 12, 9, 9, 1), ("off54", 11, 18, 18, 1), ("above54", 13, 12, 4, 3)])
def test_forms(form, logN, nq, kp, dnum):
    need_gpu()
    ks = built_lib()
    primes = _list(form, logN, nq + kp)
    p, q = primes[:kp], primes[kp:]
    P = ks.Params(logN, nq, kp, dnum, q=q, p=p)
    C = orc.Ctx(logN, nq, kp, dnum, q=q, p=p)
    P.set_bconv_tensor(True)
    for t in (0, nq - 1, nq, nq + kp - 1):
        r = (q + p)[t]
        for a in (np.full(C.N, r - 1, dtype=np.uint64), inputs.uniform_towers([r], C.N, seed=t)[0]):
            psi = orc.find_psi(r, logN)
            x = ks.to_device(a[None, :])
            P.ntt(t, x, inverse=False)
            assert np.array_equal(ks.to_host(x)[0], orc.ntt(a, logN, r, psi)), f"forward, tower {t}"
            x = ks.to_device(a[None, :])
            P.ntt(t, x, inverse=True)
            assert np.array_equal(ks.to_host(x)[0], orc.intt(a, logN, r, psi)), f"inverse, tower {t}"
    for nact in sorted({nq, max(1, nq // 2)}):
        for d in (max_y_input(C, nact), inputs.uniform_towers(C.q[:nact], C.N, seed=nact)):
            want = C.modup(nact, d)
            ext = ks.empty(want.shape)
            P.modup(nact, ks.to_device(d), ext)
            assert np.array_equal(ks.to_host(ext), want), f"ModUp, level {nact}"
        for x, cp in enumerate(max_w_cprime(C, nact)):
            out = ks.empty((nact, C.N))
            P.moddown(nact, ks.to_device(cp), out)
            assert np.array_equal(ks.to_host(out), C.moddown(nact, cp)), f"ModDown, level {nact}"
    for evk, d in ((max_evk(C), max_y_input(C, nq)), (random_evk(C, 5), inputs.uniform_towers(C.q, C.N, seed=9))):
        key = P.upload_key(evk)
        want = C.keyswitch(nq, d, evk)
        dd = ks.to_device(d)
        for df, variant, engine in ((0, 0, 1), (1, 0, 1), (2, 0, 1), (2, 2, 1), (2, 3, 1), (2, 2, 0)):
            o = ks.empty((nq, C.N)), ks.empty((nq, C.N))
            P.switch_batch_sched([(key, nq, dd, *o)], ks.Schedule(df, variant, 64, 0, 0, engine))
            for x in (0, 1):
                assert np.array_equal(ks.to_host(o[x]), want[x]), (df, variant, engine)
    assert P.device_status() == 0
