"""Tensor-core base conversion at the edges of its forms: one, two and four K
blocks (9, 18 and 36 sources), the first source past each, the CUDA-core
conversion beyond, odd target counts and target blocks, and the folding and
Montgomery epilogues (56, 54, 50 and 40-bit sets), on the largest residues."""
import numpy as np
import pytest

from oracle import oracle as orc
from paper_2311_01598_gb300 import inputs
from tests._gpu import built_lib, need_gpu, pair

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nq,kp,dnum,bits", [(9, 9, 1, 54), (10, 10, 1, 54), (18, 18, 1, 56), (19, 19, 1, 54),
                                             (36, 20, 1, 54), (37, 32, 1, 54), (20, 28, 1, 56), (40, 19, 2, 50),
                                             (8, 3, 2, 40), (33, 9, 4, 54)])
def test_conversion(nq, kp, dnum, bits):
    need_gpu()
    ks = built_lib()
    P, C = pair(11, nq, kp, dnum, bits)
    rng = np.random.Generator(np.random.PCG64(nq * kp))
    evk = np.stack([np.stack([inputs.uniform_towers(C.q + C.p, C.N, seed=int(rng.integers(1 << 30))) for _ in range(2)])
                    for _ in range(P.ndig)])
    key = P.upload_key(evk)
    for nact in sorted({nq, nq - 1, max(1, nq // 2)}):
        for d in (np.array([[q - 1] * C.N for q in C.q[:nact]], dtype=np.uint64),
                  inputs.uniform_towers(C.q[:nact], C.N, seed=nact)):
            w0, w1 = C.keyswitch(nact, d, evk)
            dd = ks.to_device(d)
            for df in ("MP", "OC"):
                o0, o1 = ks.empty((nact, C.N)), ks.empty((nact, C.N))
                P.switch(key, nact, dd, o0, o1, df)
                assert np.array_equal(ks.to_host(o0), w0) and np.array_equal(ks.to_host(o1), w1), f"{df} level {nact}"
    assert P.device_status() == 0


def test_uneven_runs():
    """A batch whose jobs' tiles cost differently (levels 1 to 24): every CTA's
    run of items starts where the one before ended."""
    need_gpu()
    ks = built_lib()
    P, C = pair(12, 24, 8, 3)
    evk = np.stack([np.stack([inputs.uniform_towers(C.q + C.p, C.N, seed=10 * j + x) for x in range(2)])
                    for j in range(P.ndig)])
    key = P.upload_key(evk)
    jobs, want = [], []
    for i, lv in enumerate([24, 1, 8, 9, 24, 2, 17, 16, 5, 24, 3]):
        d = inputs.uniform_towers(C.q[:lv], C.N, seed=100 + i)
        want.append(C.keyswitch(lv, d, evk))
        jobs.append((key, lv, ks.to_device(d), ks.empty((lv, C.N)), ks.empty((lv, C.N))))
    for sc in (ks.Schedule(2, 2, 64, 0, 0, 1), ks.Schedule(2, 1, 64, 0, 0, 1), ks.Schedule(2, 2, 64, 1, 0, 1)):
        P.switch_batch_sched(jobs, sc)
        for (_, _, _, o0, o1), (w0, w1) in zip(jobs, want):
            assert np.array_equal(ks.to_host(o0), w0) and np.array_equal(ks.to_host(o1), w1)
            o0.zero_(), o1.zero_()


@pytest.mark.parametrize("njobs,nkeys", [(2, 1), (7, 3), (64, 5), (9, 9)])
def test_shared_keys(njobs, nkeys):
    """Batches whose jobs share keys at uneven levels (the combines' job-next-to-job
    order), equal levels and the smallest ones among them."""
    need_gpu()
    ks = built_lib()
    P, C = pair(10, 7, 2, 3)
    evks = [np.stack([np.stack([inputs.uniform_towers(C.q + C.p, C.N, seed=1000 * k + 10 * j + x) for x in range(2)])
                      for j in range(P.ndig)]) for k in range(nkeys)]
    keys = [P.upload_key(e) for e in evks]
    jobs, want = [], []
    for i in range(njobs):
        lv = 1 + (5 * i + i // 4) % 7
        d = inputs.uniform_towers(C.q[:lv], C.N, seed=300 + i)
        want.append(C.keyswitch(lv, d, evks[i % nkeys]))
        jobs.append((keys[i % nkeys], lv, ks.to_device(d), ks.empty((lv, C.N)), ks.empty((lv, C.N))))
    P.switch_batch(jobs, "OC")
    for (_, _, _, o0, o1), (w0, w1) in zip(jobs, want):
        assert np.array_equal(ks.to_host(o0), w0) and np.array_equal(ks.to_host(o1), w1)


@pytest.mark.parametrize("logN,nq,kp,dnum", [(12, 3, 1, 3), (12, 9, 3, 3), (13, 7, 2, 4), (13, 9, 2, 5), (14, 8, 1, 8),
                                             (14, 9, 1, 9), (10, 12, 8, 2), (11, 5, 28, 1)])
def test_engine_by_size(logN, nq, kp, dnum):
    """Conversions on both sides of 2^17 multiply-adds: the size's engine, either
    one asked for by the schedule or the option, and the oracle agree."""
    need_gpu()
    ks = built_lib()
    P, C = pair(logN, nq, kp, dnum)
    evk = np.stack([np.stack([inputs.uniform_towers(C.q + C.p, C.N, seed=10 * j + x) for x in range(2)])
                    for j in range(P.ndig)])
    key = P.upload_key(evk)
    for nact in (nq, 1):
        d = inputs.uniform_towers(C.q[:nact], C.N, seed=nact)
        want = C.keyswitch(nact, d, evk)
        dd = ks.to_device(d)
        for option in (None, True, False):
            if option is not None:
                P.set_bconv_tensor(option)
            for df in (0, 1, 2):
                for engine in (-1, 0, 1):
                    o = ks.empty((nact, C.N)), ks.empty((nact, C.N))
                    P.switch_batch_sched([(key, nact, dd, *o)], ks.Schedule(df, 2, 64, 0, -1, engine))
                    for x in (0, 1):
                        assert np.array_equal(ks.to_host(o[x]), want[x]), (option, df, engine, nact)
    assert P.device_status() == 0
