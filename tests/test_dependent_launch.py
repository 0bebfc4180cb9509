"""Dependent launches: a kernel of a stream's chain may start before the one
ahead of it is complete, and only its wait orders it.  A launch whose blocks
all left without waiting would be complete before its predecessor, and the
kernel after it would start on data still being written.  On the CPU: in the
sources, every path out of such a kernel passes its wait, but for a transform's
blocks of bypassed limbs, whose launchers make sure of others.  On the GPU: the calls
that would have launches without any work (the fused variant's Q section with one
active digit, a tower shard inside one digit) queue nothing for them and agree with the
oracle."""
import glob
import os
import re

import numpy as np
import pytest

from paper_2311_01598_gb300 import inputs
from tests._gpu import built_lib, need_gpu, pair

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2311_01598_gb300", "csrc")


def _kernels():
    """name -> body of every __global__ function, comments removed."""
    out = {}
    for f in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        text = re.sub(r"//[^\n]*|/\*.*?\*/", "", open(f).read(), flags=re.S)
        for m in re.finditer(r"__global__[^{;]*?\b(k_\w+)\s*\([^{;]*\)\s*\{", text):
            depth, at = 1, m.end()
            while depth:
                depth += {"{": 1, "}": -1}.get(text[at], 0)
                at += 1
            out[m.group(1)] = text[m.end():at - 1]
    return out


def test_every_path_waits():
    kernels = _kernels()
    dependent = {k for k, body in kernels.items() if "pdl_start();" in body}
    starts = sum(open(f).read().count("pdl_start();") for f in glob.glob(os.path.join(CSRC, "*.cu")))
    assert len(dependent) == starts >= 15  # the scan found them all
    for k in sorted(dependent):
        body = kernels[k]
        wait = re.search(r"(?<!return )\bpdl_wait\(\);", body)
        assert wait, f"{k} never waits"
        head = body[:wait.start()].replace("if (L.skip) return;", "")
        assert not re.search(r"\breturn\b(?!\s*pdl_wait\(\);)", head), f"{k} may leave before its wait"


def test_launched_kernels_wait():
    """Only kernels with a wait are launched as dependent ones."""
    kernels = _kernels()
    launched = set()
    for f in glob.glob(os.path.join(CSRC, "*.cu")):
        launched |= set(re.findall(r"launch_(?:dep\(st,|cluster\()\s*(k_\w+)", open(f).read()))
    assert len(launched) >= 15
    for k in sorted(launched):
        assert "pdl_start();" in kernels[k] and "pdl_wait();" in kernels[k], k


@pytest.mark.gpu
@pytest.mark.parametrize("logN,nq,kp,dnum,nact", [(10, 4, 2, 1, 4), (12, 6, 2, 3, 2), (13, 3, 3, 1, 2), (16, 8, 8, 1, 8),
                                                  (16, 9, 3, 3, 3), (17, 4, 4, 1, 3)])
def test_fused_one_digit(logN, nq, kp, dnum, nact):
    """The fused variant where every Q tower lies in the only active digit: alone,
    and beside a job with more digits (whose conversion is then launched)."""
    need_gpu()
    ks = built_lib()
    P, C = pair(logN, nq, kp, dnum)
    evk = np.stack([np.stack([inputs.uniform_towers(C.q + C.p, C.N, seed=10 * j + x) for x in range(2)])
                    for j in range(P.ndig)])
    key = P.upload_key(evk)
    levels = [nact] * 3 + ([nq] if dnum > 1 else [])
    jobs, want = [], []
    for i, lv in enumerate(levels):
        d = inputs.uniform_towers(C.q[:lv], C.N, seed=40 + i)
        want.append(C.keyswitch(lv, d, evk))
        jobs.append((key, lv, ks.to_device(d), ks.empty((lv, C.N)), ks.empty((lv, C.N))))
    for engine in (-1, 0, 1):
        sc = ks.Schedule(2, 0, 64, 0, 0, engine)
        for n in sorted({1, 3, len(jobs)}):
            before = ks.kernel_launches()
            P.switch_batch_sched(jobs[:n], sc)
            # iNTT 2, P section: conversion, column, row, inverse column; Q section:
            # conversion (with more than one digit), ModDown's, column, row
            assert ks.kernel_launches() - before == (9 if n < 4 else 10)
            for (_, _, _, o0, o1), (w0, w1) in zip(jobs[:n], want):
                assert np.array_equal(ks.to_host(o0), w0) and np.array_equal(ks.to_host(o1), w1), (engine, n)
                o0.zero_(), o1.zero_()


@pytest.mark.gpu
@pytest.mark.parametrize("logN,nq,dnum,nact", [(12, 6, 1, 6), (14, 6, 2, 3), (16, 6, 1, 5)])
def test_shard_inside_one_digit(logN, nq, dnum, nact):
    """A rank without special towers whose Q towers are all of the active digit's:
    its conversion and its forward transforms have nothing to do."""
    torch = need_gpu()
    ks = built_lib()
    from paper_2311_01598_gb300 import dist as kd
    P, C = pair(logN, nq, 2, dnum)
    evk = np.stack([np.stack([inputs.uniform_towers(C.q + C.p, C.N, seed=10 * j + x) for x in range(2)])
                    for j in range(P.ndig)])
    key = P.upload_key(evk)
    parts = [(0, nq // 2, 0, 0), (nq // 2, nq, 0, 2)]
    skeys = [P.key_shard(key, ks.Shard(*pt)) for pt in parts]
    d = inputs.uniform_towers(C.q[:nact], C.N, seed=7)
    ranges = [kd.active_q(pt, nact) for pt in parts]
    d_own = [ks.to_device(np.ascontiguousarray(d[a:b])) if b > a else ks.empty((0, C.N)) for a, b in ranges]
    outs = kd.sharded_keyswitch(P, skeys, parts, nact, d_own, gather_y=lambda ys: torch.cat(ys, dim=0),
                                gather_w=lambda ws: torch.cat(ws, dim=1))
    want = C.keyswitch(nact, d, evk)
    for x in range(2):
        got = np.concatenate([ks.to_host(o[x]) for o in outs if o[x].shape[0] > 0])
        assert np.array_equal(got, want[x])
    a, b = ranges[0]  # the first rank's key product is its only launch
    y = ks.empty((nact, C.N))
    cp = ks.empty((2, b - a, C.N))
    scratch = ks.empty((P.shard_scratch_words(ks.Shard(*parts[0]), nact),))
    before = ks.kernel_launches()
    P.shard_keyprod(skeys[0], nact, y, d_own[0], cp, scratch)
    assert ks.kernel_launches() - before == 1


@pytest.mark.gpu
@pytest.mark.parametrize("logN,nq,kp", [(10, 48, 17), (13, 7, 2), (14, 60, 32), (16, 34, 4), (17, 3, 2)])
def test_transforms_alone(logN, nq, kp):
    """Transforms called one after the other on the same limbs, below, at and past
    the sizes where the next kernel may start with a pass (2^16 words; a wave, half
    a wave of blocks): inverse of forward, and forward three times, against the
    oracle on the first and the last limb."""
    need_gpu()
    ks = built_lib()
    from oracle import oracle as orc
    P, C = pair(logN, nq, kp, 1)
    primes = P.q + P.p
    nt = len(primes)
    a = inputs.uniform_towers(primes, C.N, seed=logN)
    words = 1 << 16 >> logN
    counts = {1, words, words + 1, nt - 1, nt}
    for waves in (8 * 152, 16 * 152):  # row blocks of half a wave and of one
        rows = 4 if logN >= 16 else 8
        limbs = waves // ((1 << logN - logN // 2) // rows)
        counts |= {limbs, limbs + 1}
    for n in sorted(c for c in counts if 1 <= c <= nt):
        x = ks.to_device(a[:n])
        for _ in range(2):
            P.ntt(0, x, inverse=False)
            P.ntt(0, x, inverse=True)
        assert np.array_equal(ks.to_host(x), a[:n]), n
        for _ in range(3):
            P.ntt(0, x, inverse=False)
        got = ks.to_host(x)
        for t in {0, n - 1}:
            want = a[t]
            for _ in range(3):
                want = orc.ntt(want, logN, primes[t], orc.find_psi(primes[t], logN))
            assert np.array_equal(got[t], want), (n, t)


@pytest.mark.gpu
@pytest.mark.parametrize("cluster", [1, 2])
@pytest.mark.parametrize("logN,nq,kp", [(10, 48, 17), (14, 60, 32), (16, 40, 4)])
def test_cluster_transforms_alone(logN, nq, kp, cluster):
    """The same for the one-launch cluster form, below and past 2^16 words and a
    wave of blocks (16 CTAs a limb at 2^16, 4 or 8 at 2^14, 1 or 2 at 2^10)."""
    need_gpu()
    ks = built_lib()
    from oracle import oracle as orc
    P, C = pair(logN, nq, kp, 1)
    P.set_ntt_cluster(cluster)
    primes = P.q + P.p
    a = inputs.uniform_towers(primes, C.N, seed=logN)
    for n in sorted({1, 2, min(64, len(primes)), 19, 38, len(primes)}):
        x = ks.to_device(a[:n])
        for _ in range(2):
            P.ntt(0, x, inverse=False)
            P.ntt(0, x, inverse=True)
        assert np.array_equal(ks.to_host(x), a[:n]), n
        for _ in range(2):
            P.ntt(0, x, inverse=False)
        got = ks.to_host(x)
        for t in {0, n - 1}:
            psi = orc.find_psi(primes[t], logN)
            assert np.array_equal(got[t], orc.ntt(orc.ntt(a[t], logN, primes[t], psi), logN, primes[t], psi)), (n, t)
