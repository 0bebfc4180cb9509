"""The combine kernels' job-next-to-job order, taken by batches that share keys
and read more than L2 holds: on both sides of that line, uneven levels, the
smallest ones among them, one key to all different.  Equal to the jobs switched
one by one under the max-parallel dataflow; the first one to the oracle too."""
import numpy as np
import pytest

from oracle import oracle as orc
from paper_2311_01598_gb300 import inputs
from tests._gpu import built_lib, need_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("logN,nq,kp,dnum,levels,nkeys", [
    (16, 24, 8, 3, [24, 24], 1), (16, 24, 8, 3, [24, 1, 17, 24, 9], 3), (16, 24, 8, 3, [1, 2, 24, 24, 8, 16, 1], 6),
    (14, 10, 4, 3, [10] * 12, 2), (14, 10, 4, 3, [10] * 13, 2),  # 2^14: the line lies between 12 and 13 jobs
    (14, 10, 4, 3, [1 + (7 * i + i // 3) % 10 for i in range(64)], 5), (17, 9, 3, 3, [9, 4, 1, 7, 9], 2),
    (16, 6, 1, 6, [6, 6, 1, 5, 3, 6, 2, 6, 6], 4)])
def test_shared_order(logN, nq, kp, dnum, levels, nkeys):
    torch = need_gpu()
    ks = built_lib()
    P = ks.Params(logN, nq, kp, dnum)
    P.set_batch_lanes(1)
    C = orc.Ctx(logN, nq, kp, dnum)
    evk = np.stack([np.stack([inputs.uniform_towers(C.q + C.p, C.N, seed=10 * j + x) for x in range(2)])
                    for j in range(P.ndig)])
    keys = [P.upload_key(evk)] + [P.key_synthetic(i) for i in range(1, nkeys)]
    ds = [inputs.uniform_towers(C.q[:lv], C.N, seed=100 + i) if i == 0 else None for i, lv in enumerate(levels)]
    gen = torch.Generator(device="cuda")
    gen.manual_seed(1)
    jobs, want = [], []
    for i, lv in enumerate(levels):
        d = ks.to_device(ds[0]) if i == 0 else torch.stack(
            [torch.randint(0, q, (P.N,), generator=gen, device="cuda", dtype=torch.int64) for q in P.q[:lv]])
        jobs.append((keys[i % nkeys], lv, d, ks.empty((lv, P.N)), ks.empty((lv, P.N))))
        a, b = ks.empty((lv, P.N)), ks.empty((lv, P.N))
        P.switch(jobs[-1][0], lv, d, a, b, "MP")
        want.append((a, b))
    w0, w1 = C.keyswitch(levels[0], ds[0], evk)
    assert np.array_equal(ks.to_host(want[0][0]), w0) and np.array_equal(ks.to_host(want[0][1]), w1)
    for sc in (ks.Schedule(2, 2, 64, 0, 0, -1), ks.Schedule(2, 1, 64, 1, 0, -1), ks.Schedule(2, 2, 4, 0, 0, -1)):
        P.switch_batch_sched(jobs, sc)
        for (_, _, _, o0, o1), (a, b) in zip(jobs, want):
            assert torch.equal(o0, a) and torch.equal(o1, b)
            o0.zero_(), o1.zero_()
