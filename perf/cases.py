"""Performance cases: the calls a user of the key-switching library makes, over the sizes they are made at.

A case is a dict of plain values.  Its "op" says which public entry point runs:

  switch    one ciphertext (Params.switch) under a dataflow
  batch     many ciphertexts at uneven levels (Params.switch_batch, or
            switch_batch_sched when the case fixes a schedule)
  hoisted   several rotations of one ciphertext sharing one ModUp
            (switch_hoisted) and the rotated first component (automorph)
  ntt       forward or inverse negacyclic NTT of a set of towers
  host      a batch whose ciphertexts live in pinned host memory
            (switch_batch_host): copies in, key switches, copies out

Parameter sets (prime tables on the device) are kept between preparations, as a program keeps them for its
whole life; keys, ciphertexts and output buffers belong to one state.  Keys are uniform words (a real key
is computationally indistinguishable from them and the arithmetic does not depend on the values), except
compressed keys, which are generated.
"""
import collections

import numpy as np
import torch

from paper_2311_01598_gb300 import ks

_DEVICE = "cuda"
_params = collections.OrderedDict()  # parameter sets in use, newest last


def listed():
    return [
        # a small ring (tests and smoke set): one key switch is a dozen launches of a few microseconds each
        dict(name="switch_n12", op="switch", logN=12, nq=3, kp=1, dnum=3, bits=50, level=3, dataflow="OC"),
        # the benchmark's parameter set, one ciphertext at the top level: the latency of a lone rotation or
        # relinearisation in an interactive program
        dict(name="switch_n16", op="switch", logN=16, nq=24, kp=8, dnum=3, bits=54, level=24, dataflow="OC"),
        # the paper's ARK set under the digit-centric dataflow, one level down: a ragged last digit
        dict(name="switch_n16_ark_dc", op="switch", logN=16, nq=24, kp=6, dnum=4, bits=54, level=23, dataflow="DC"),
        # the paper's BTS3 set (bootstrapping scale, N = 2^17): the largest single key switch, 360 MB of key
        dict(name="switch_n17_bts3", op="switch", logN=17, nq=45, kp=15, dnum=3, bits=54, level=45, dataflow="OC"),
        # the paper's BTS1 set under the max-parallel dataflow: one digit, more sources than the tensor-core base
        # conversion takes
        dict(name="switch_n17_bts1_mp", op="switch", logN=17, nq=28, kp=28, dnum=1, bits=54, level=28, dataflow="MP"),
        # the benchmark step: 16 ciphertexts, a key each, under the schedule the autotuner picks for it
        dict(name="batch16_n16", op="batch", logN=16, nq=24, kp=8, dnum=3, bits=54, jobs=16, keys=16, lmin=24,
             lmax=24, sched="2,2,64,0,0,1", compressed=False),
        # a busy evaluator: 64 ciphertexts at levels 4..24, 16 rotation keys, no tuning done
        dict(name="batch64_mixed_n16", op="batch", logN=16, nq=24, kp=8, dnum=3, bits=54, jobs=64, keys=16, lmin=4,
             lmax=24, sched="", compressed=False),
        # compressed keys (half of the key regenerated from a seed) at a middle ring degree
        dict(name="batch6_n14_compressed", op="batch", logN=14, nq=10, kp=4, dnum=3, bits=54, jobs=6, keys=3, lmin=5,
             lmax=10, sched="", compressed=True),
        # eight rotations of one ciphertext, as in a matrix-vector product or a slot sum
        dict(name="hoisted8_n16", op="hoisted", logN=16, nq=24, kp=8, dnum=3, bits=54, level=24, rot=8),
        # transforms called alone, by programs that compose their own schedules: every tower of a set, and few
        dict(name="ntt_fwd_n16", op="ntt", logN=16, nq=24, kp=8, dnum=3, bits=54, first=0, towers=32, inverse=False),
        dict(name="ntt_inv_n13", op="ntt", logN=13, nq=6, kp=2, dnum=3, bits=56, first=1, towers=5, inverse=True),
        # ciphertexts in host memory: what a program pays end to end
        dict(name="host12_n16", op="host", logN=16, nq=24, kp=8, dnum=3, bits=54, jobs=12, keys=4, lmin=11, lmax=17,
             dataflow="OC"),
    ]


def draw(rng):
    most = max(_cost(c) for c in listed())
    while True:
        op = rng.choice(["switch", "switch", "batch", "batch", "hoisted", "ntt", "host"])
        logN = rng.randint(11, 17)
        nq = min(45, max(2, round(2 ** rng.uniform(1, 5.5))))
        dnum = rng.randint(1, min(nq, 6))
        alpha = -(-nq // dnum)
        kp = max(1, min(28, alpha + rng.randint(-1, 1)))
        c = dict(op=op, logN=logN, nq=nq, kp=kp, dnum=dnum, bits=rng.choice([50, 54, 54, 56]))
        if op == "switch":
            c.update(level=rng.randint(1, nq), dataflow=rng.choice(["OC", "OC", "MP", "DC"]))
        elif op == "batch":
            lmin = rng.randint(1, nq)
            sched = rng.choice(["", "", "2,2,64,0,0,1", "2,2,16,2,0,1", "2,1,64,1,0,0"])
            c.update(jobs=max(2, round(2 ** rng.uniform(1, 6))), keys=rng.randint(1, 8), lmin=lmin,
                     lmax=rng.randint(lmin, nq), sched=sched, compressed=logN <= 14 and nq <= 12 and rng.random() < 0.3)
        elif op == "hoisted":
            c.update(level=rng.randint(1, nq), rot=rng.randint(2, 12))
        elif op == "ntt":
            first = rng.randint(0, nq + kp - 1)
            c.update(first=first, towers=rng.randint(1, nq + kp - first), inverse=rng.random() < 0.5)
        else:
            lmin = rng.randint(1, nq)
            c.update(jobs=rng.randint(1, 12), keys=rng.randint(1, 4), lmin=lmin, lmax=rng.randint(lmin, nq),
                     dataflow="OC")
        if _cost(c) <= most and _memory(c) <= 12e9:
            return c


# ---------------------------------------------------------------- state
def _set(c):
    """The parameter set of a case (the few most recent ones are kept)."""
    k = (c["logN"], c["nq"], c["kp"], c["dnum"], c["bits"])
    if k in _params:
        _params.move_to_end(k)
    else:
        _params[k] = ks.Params(c["logN"], c["nq"], c["kp"], c["dnum"], prime_bits=c["bits"])
        while len(_params) > 6:
            _params.popitem(last=False)
    return _params[k]


def _levels(c):
    """Levels of the jobs: a fixed mix over [lmin, lmax], the same for every seed."""
    span = c["lmax"] - c["lmin"] + 1
    return [c["lmin"] + (7 * i + i // 3) % span for i in range(c["jobs"])]


def _uniform(primes, N, gen):
    """[towers][N] residues, row t uniform below primes[t]."""
    out = torch.empty((len(primes), N), dtype=torch.int64, device=_DEVICE)
    for t, q in enumerate(primes):
        torch.randint(0, int(q), (N,), generator=gen, device=_DEVICE, out=out[t])
    return out


def _keys(P, count, seed, compressed):
    if not compressed:
        return [P.key_synthetic(seed * 1000 + i) for i in range(count)]
    r = np.random.default_rng(seed)
    s = r.integers(-1, 2, P.N).astype(np.int8)
    return [P.keygen_compressed(s, r.integers(-1, 2, P.N).astype(np.int64), seed * 1000 + i) for i in range(count)]


def prepare(case, seed):
    c = case
    P = _set(c)
    gen = torch.Generator(device=_DEVICE)
    gen.manual_seed(seed)
    st = {"op": c["op"], "P": P}
    if c["op"] == "ntt":
        primes = (P.q + P.p)[c["first"]:c["first"] + c["towers"]]
        st.update(x=_uniform(primes, P.N, gen), first=c["first"], inverse=c["inverse"])
    elif c["op"] == "switch":
        lv = c["level"]
        st.update(key=_keys(P, 1, seed, False)[0], level=lv, d=_uniform(P.q[:lv], P.N, gen),
                  out=(ks.empty((lv, P.N)), ks.empty((lv, P.N))), dataflow=c["dataflow"])
    elif c["op"] == "hoisted":
        lv, R = c["level"], c["rot"]
        st.update(keys=_keys(P, R, seed, False), level=lv, c0=_uniform(P.q[:lv], P.N, gen),
                  d=_uniform(P.q[:lv], P.N, gen), galois=[pow(5, 3 * r + 1, 2 * P.N) for r in range(R)],
                  rot0=ks.empty((R, lv, P.N)), out=(ks.empty((R, lv, P.N)), ks.empty((R, lv, P.N))))
    else:
        host = c["op"] == "host"
        levels = _levels(c)
        keys = _keys(P, c["keys"], seed, c.get("compressed", False))
        rows = sum(levels)
        d = torch.cat([_uniform(P.q[:lv], P.N, gen) for lv in levels])
        if host:
            d = d.cpu().pin_memory()
            o0, o1 = (torch.empty((rows, P.N), dtype=torch.int64, pin_memory=True) for _ in range(2))
        else:
            o0, o1 = ks.empty((rows, P.N)), ks.empty((rows, P.N))
        jobs, at = [], 0
        for i, lv in enumerate(levels):
            jobs.append((keys[i % len(keys)], lv, d[at:at + lv], o0[at:at + lv], o1[at:at + lv]))
            at += lv
        sched = c.get("sched", "")
        st.update(jobs=jobs, out=(o0, o1), sched=ks.Schedule(*map(int, sched.split(","))) if sched else None)
    return st


def run(state):
    s = state
    P, op = s["P"], s["op"]
    if op == "ntt":
        # in place on the program's buffer: every pass transforms what the last one left, as canonical as the first
        P.ntt(s["first"], s["x"], s["inverse"])
        return s["x"]
    if op == "switch":
        P.switch(s["key"], s["level"], s["d"], *s["out"], s["dataflow"])
        return s["out"]
    if op == "hoisted":
        o0, o1, r0 = s["out"][0], s["out"][1], s["rot0"]
        P.switch_hoisted(s["keys"], s["galois"], s["level"], s["d"], list(o0), list(o1))
        for r, g in enumerate(s["galois"]):
            P.automorph(0, g, s["c0"], r0[r])
        return o0, o1, r0
    if op == "host":
        P.switch_batch_host(s["jobs"], "OC")
        return s["out"]
    if s["sched"] is not None:
        P.switch_batch_sched(s["jobs"], s["sched"])
    else:
        P.switch_batch(s["jobs"], "OC")
    return s["out"]


# ---------------------------------------------------------------- work
def _switch_ops(c, lv):
    """(key bytes, NTT limbs, base-conversion products per coefficient, key products per coefficient) of one key
    switch at level lv."""
    alpha = -(-c["nq"] // c["dnum"])
    nd = -(-lv // alpha)
    own = [min(alpha, lv - j * alpha) for j in range(nd)]
    up = [lv + c["kp"] - a for a in own]  # towers digit j is raised to
    key = nd * 2 * (lv + c["kp"])         # limbs of the key that level lv reads
    ntt = lv + sum(up) + 2 * c["kp"] + 2 * lv
    conv = sum(a * u for a, u in zip(own, up)) + 2 * c["kp"] * lv
    return key, ntt, conv, key


def work(case):
    """Bytes: every input and key limb read once, every output limb written once.  Operations: two (a modular
    multiplication and an addition) per butterfly, base-conversion term and key product."""
    c = case
    N = 1 << c["logN"]
    limb = 8 * N
    if c["op"] == "ntt":
        return {"bytes": 2 * c["towers"] * limb, "flops": 2 * c["towers"] * (N // 2) * c["logN"]}
    if c["op"] == "hoisted":
        lv, R = c["level"], c["rot"]
        key, ntt, conv, mac = _switch_ops(c, lv)
        alpha = -(-c["nq"] // c["dnum"])
        raised = ntt - 2 * c["kp"] - 2 * lv
        down = 2 * c["kp"] + 2 * lv
        nd = -(-lv // alpha)
        up_conv = conv - 2 * c["kp"] * lv
        limbs = 2 * lv + R * (key * (1 if nd else 0) + 3 * lv)
        ops = (raised + R * down) * (N // 2) * c["logN"] + (up_conv + R * (2 * c["kp"] * lv + mac)) * N
        return {"bytes": limbs * limb, "flops": 2 * ops}
    levels = _levels(c) if c["op"] in ("batch", "host") else [c["level"]]
    read, bfly, mul = 0, 0, 0
    top = {}  # highest level each key is used at: its limbs are read once
    for i, lv in enumerate(levels):
        key, ntt, conv, mac = _switch_ops(c, lv)
        k = i % c.get("keys", 1)
        half = 2 if not c.get("compressed", False) else 1
        top[k] = max(top.get(k, 0), key * half // 2)
        read += 3 * lv
        bfly += ntt * (N // 2) * c["logN"]
        mul += (conv + mac) * N
    return {"bytes": (read + sum(top.values())) * limb, "flops": 2 * (bfly + mul)}


def _cost(c):
    w = work(c)
    # seconds at about the rates of the path: memory, integer multiplications, and the host link for host jobs
    extra = 0
    if c["op"] == "host":
        extra = 3 * sum(_levels(c)) * (8 << c["logN"]) / 1e11
    return w["bytes"] / 5e12 + w["flops"] / 1.2e12 + extra


def _memory(c):
    """Bytes of one state and of the library's scratch for it, roughly."""
    N8 = 8 << c["logN"]
    nt = c["nq"] + c["kp"]
    alpha = -(-c["nq"] // c["dnum"])
    nd = -(-c["nq"] // alpha)
    jobs = c.get("jobs", c.get("rot", 1))
    keys = c.get("keys", c.get("rot", 1))
    return N8 * (keys * nd * 2 * nt + jobs * (nd * nt + 10 * c["nq"]))


# ---------------------------------------------------------------- exact values
def _bitrev(n, bits):
    r = np.zeros(n, dtype=np.int64)
    for b in range(bits):
        r |= ((np.arange(n) >> b) & 1) << (bits - 1 - b)
    return r


def _psi(q, N):
    """The primitive 2N-th root the library fixes: x^((q-1)/2N) for the least x >= 2 that gives one."""
    x = 2
    while True:
        r = pow(x, (q - 1) // (2 * N), q)
        if pow(r, N, q) == q - 1:
            return r
        x += 1


def _ntt_exact(a, q, logN, inverse):
    """Negacyclic NTT of one tower with Python integers: slot k holds the value at psi^(2*brv(k)+1)."""
    N = 1 << logN
    psi = _psi(q, N)
    powers = np.empty(N, dtype=object)
    v = 1
    for i in range(N):
        powers[i] = v
        v = v * psi % q
    rev = _bitrev(N, logN)
    if not inverse:
        x = a.astype(object) * powers % q  # twist, then a cyclic transform of length N at omega = psi^2
        w0 = psi * psi % q
        y = _cyclic(x, q, w0, logN, rev)   # natural order
        return y[rev]
    w0 = pow(psi, -2, q)
    y = _cyclic(a.astype(object)[rev], q, w0, logN, rev)
    ninv = pow(N, -1, q)
    inv = np.empty(N, dtype=object)
    v, ip = ninv, pow(psi, -1, q)
    for i in range(N):
        inv[i] = v
        v = v * ip % q
    return y * inv % q


def _cyclic(x, q, w, logN, rev):
    N = 1 << logN
    x = x[rev].copy()
    for s in range(logN):
        h = 1 << s
        ws = pow(w, N >> (s + 1), q)
        tw = np.empty(h, dtype=object)
        v = 1
        for i in range(h):
            tw[i] = v
            v = v * ws % q
        x = x.reshape(-1, 2, h)
        t = x[:, 1, :] * tw % q
        x = np.stack([(x[:, 0, :] + t) % q, (x[:, 0, :] - t) % q], axis=1).reshape(N)
    return x


def exact(case, seed):
    """What one pass gives, with Python integers, for transforms small enough; None elsewhere (all outputs are
    integers)."""
    c = case
    if c["op"] != "ntt" or c["towers"] << c["logN"] > 1 << 20:
        return None
    st = prepare(c, seed)
    x = st["x"].cpu().numpy()
    primes = (st["P"].q + st["P"].p)[c["first"]:c["first"] + c["towers"]]
    rows = [_ntt_exact(x[t], int(q), c["logN"], c["inverse"]) for t, q in enumerate(primes)]
    return torch.from_numpy(np.stack([np.array(r.tolist(), dtype=np.int64) for r in rows]))
