"""A batch over stream lanes: which jobs share a lane, and so the scratch a lane
holds, follows from the jobs' order and levels, not from which keys they use.
A batch of a shape that has run before allocates nothing and can be captured
with keys the parameter set has not been called with."""
import numpy as np
import pytest

from tests._gpu import built_lib, need_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sched", [None, (2, 2, 64, 0, 0, 1), (2, 2, 3, 0, -1, -1)])
@pytest.mark.parametrize("lanes", [2, 4])
def test_other_keys_same_lanes(sched, lanes):
    torch = need_gpu()
    ks = built_lib()
    P = ks.Params(13, 24, 8, 3)
    P.set_batch_lanes(lanes)
    levels = [24, 2] * 8  # a lane of the small ones alone needs a tenth of the scratch
    keys = sorted((P.key_synthetic(i) for i in range(8)), key=lambda k: k.handle)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(3)
    data = []
    for lv in levels:
        d = torch.stack([torch.randint(0, q, (P.N,), generator=gen, device="cuda", dtype=torch.int64) for q in P.q[:lv]])
        data.append((lv, d, ks.empty((lv, P.N)), ks.empty((lv, P.N))))

    def batch(pick):
        return [(keys[pick(i // 2, lv)], lv, d, o0, o1) for i, (lv, d, o0, o1) in enumerate(data)]

    spread = batch(lambda i, lv: i)                                    # every key at both levels
    bylevel = batch(lambda i, lv: i // 2 if lv == 24 else 4 + i // 2)  # each key at one level

    def run(jobs, st):
        if sched is None:
            P.switch_batch(jobs, "OC", st)
        else:
            P.switch_batch_sched(jobs, ks.Schedule(*sched), st)

    st = torch.cuda.Stream()
    with torch.cuda.stream(st):
        run(spread, st)
        run(spread, st)
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    with torch.cuda.stream(st):
        run(bylevel, st)
    torch.cuda.synchronize()
    assert torch.cuda.mem_get_info()[0] == free, "the batch took memory for other keys"

    P.set_batch_lanes(1)
    want = []
    for key, lv, d, o0, o1 in spread:
        a, b = ks.empty((lv, P.N)), ks.empty((lv, P.N))
        P.switch(key, lv, d, a, b, "MP")
        want.append((a, b))
    P.set_batch_lanes(lanes)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=st):
        run(spread, st)
    for _, _, o0, o1 in data:
        o0.zero_(), o1.zero_()
    g.replay()
    torch.cuda.synchronize()
    for (a, b), (_, _, o0, o1) in zip(want, data):
        assert torch.equal(a, o0) and torch.equal(b, o1)
    fresh = [(k2, *j[1:]) for k2, j in zip([P.key_synthetic(100 + i) for i in range(16)], spread)]
    torch.cuda.synchronize()
    g2 = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g2, stream=st):
        run(fresh, st)
    g2.replay()
    torch.cuda.synchronize()
    for (key, lv, d, o0, o1), x in zip(fresh, range(16)):
        a, b = ks.empty((lv, P.N)), ks.empty((lv, P.N))
        P.switch(key, lv, d, a, b, "MP")
        assert torch.equal(a, o0) and torch.equal(b, o1), x
