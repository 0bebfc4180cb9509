"""The autotuner and schedules that run the same launches: the split variant
always, the fused and the per-tower one for compressed keys, the per-tower one
where the ring has no cluster form.  They take their twin's time and are never
picked, so that a pick means the same for every later batch of its signature."""
import pytest

from paper_2311_01598_gb300 import inputs
from tests._gpu import built_lib, need_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("logN,kinds", [(12, "cccc"), (13, "cccc"), (12, "ffff"), (13, "ffff"), (12, "cffc"), (14, "ccccccccc")])
def test_twins(logN, kinds):
    need_gpu()
    ks = built_lib()
    P = ks.Params(logN, 6, 2, 3)
    s = inputs.ternary_secret(P.N, 3)
    sp = inputs.galois_secret(s, 5)
    keys = {"c": P.keygen_compressed(s, sp, seed=1), "f": P.key_synthetic(1)}
    jobs = [(keys[k], 6, ks.to_device(inputs.uniform_towers(P.q, P.N, seed=i)), ks.empty((6, P.N)), ks.empty((6, P.N)))
            for i, k in enumerate(kinds)]
    best, ms = P.autotune(jobs, reps=2)
    c = P.tune_candidates()
    at = {t.as_tuple(): i for i, t in enumerate(c)}
    assert len(ms) == len(c) and all(0 < m < 1e3 for m in ms)
    same = {1}
    if "f" not in kinds:
        same |= {0, 3}
    elif logN == 13:  # no cluster geometry
        same.add(3)
    for i, t in enumerate(c):
        df, v, chunk, order = t.as_tuple()
        if df == 2 and v in same:
            assert ms[i] == ms[at[(2, 2, chunk, order)]], t
    assert best.as_tuple() in at and not (best.dataflow == 2 and best.oc_variant in same), best
    assert P.tune_cache_get(len(jobs), 6).as_tuple() == best.as_tuple()
