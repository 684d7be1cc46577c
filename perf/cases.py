"""The work a user of the library has it do, as cases that can be timed and compared.

Kinds of case:
  ntt        one transform on device vectors through Plan.execute: forward,
             inverse and coset, three scalar fields, tables precomputed or
             formed on the fly, 2^12 (a single small call, launches count) to
             2^26 (the largest configured size); odd logarithms among them
  host       the same from pinned host memory and back (Plan.execute_host)
  groth16    the Groth16 H sequence: a graph replayed on fixed buffers, or the
             call on the caller's buffers
  batch      uneven independent transforms of two fields in one call
  pointwise  (a b - c) z over a vector of any length, the step between the
             coset transforms of a prover that runs them one by one
"""
import math
import random

import numpy as np
import torch

import paper_2509_22684_gb300 as zk

# scalar fields: modulus, multiplicative generator, 2-adicity of modulus - 1
FIELDS = {
    "bls12_381_fr": (0x73eda753299d7d483339d80809a1d80553bda402fffe5bfeffffffff00000001, 7, 32),
    "bn254_fr": (0x30644e72e131a029b85045b68181585d2833e84879b9709143e1f593f0000001, 5, 28),
    "bls12_377_fr": (0x12ab655e9a2ca55660b44d1e5c37b00159aa76fed00000010a11800000000001, 22, 47),
}
# transforms up to this size have a plain big-integer statement that ends in seconds
EXACT_LOG_N = 17


def listed():
    return [
        # the smallest single call: two short launches
        _ntt("single_2e12", "bls12_381_fr", 12),
        # small prover circuits, an inverse transform
        _ntt("inverse_2e16", "bn254_fr", 16, inverse=True),
        # an odd logarithm on the third field, coset input scale
        _ntt("coset_2e17", "bls12_377_fr", 17, coset=True),
        # mid-size circuit, the last transform of a quotient computation
        _ntt("coset_inverse_2e20", "bls12_381_fr", 20, inverse=True, coset=True),
        # device memory is short: twiddles formed on the fly
        _ntt("on_the_fly_2e22", "bn254_fr", 22, twiddle="otf"),
        # the size the library's headline figure is quoted on
        _ntt("single_2e24", "bls12_381_fr", 24),
        # the largest configured transform
        _ntt("inverse_2e26", "bls12_381_fr", 26, inverse=True),
        # the transform as a host program sees it, copies included
        dict(name="host_2e20", kind="host", field="bls12_381_fr", log_n=20, inverse=False),
        # small circuits proved in a loop: one captured graph, replayed
        dict(name="groth16_graph_2e14", kind="groth16", field="bn254_fr", log_n=14, graph=True),
        # a production circuit, called on the prover's own buffers
        dict(name="groth16_2e22", kind="groth16", field="bls12_381_fr", log_n=22, graph=False),
        # 64 transforms of uneven sizes and two fields, as a server batches them
        dict(name="batch_64", kind="batch", jobs=64, low=10, high=20, mix=4000),
        # the pointwise step alone, over a length that is no power of two
        dict(name="pointwise_3000001", kind="pointwise", field="bls12_381_fr", n=3000001),
    ]


def _ntt(name, field, log_n, inverse=False, coset=False, twiddle="auto"):
    return dict(name=name, kind="ntt", field=field, log_n=log_n, inverse=inverse, coset=coset,
                twiddle=twiddle)


def draw(rng):
    kind = rng.choice(["ntt", "ntt", "ntt", "ntt", "host", "groth16", "batch", "pointwise"])
    field = rng.choice(sorted(FIELDS))
    if kind == "ntt":
        c = _ntt("", field, rng.randint(10, 26 if field != "bls12_377_fr" else 25),
                 rng.random() < 0.5, rng.random() < 0.4, "otf" if rng.random() < 0.25 else "auto")
        # the largest listed transform is the plain 2^26 one with tables
        if c["log_n"] == 26 and (c["coset"] or c["twiddle"] == "otf"):
            c["log_n"] = 25
        del c["name"]
        return c
    if kind == "host":
        return dict(kind=kind, field=field, log_n=rng.randint(12, 23), inverse=rng.random() < 0.5)
    if kind == "groth16":
        return dict(kind=kind, field=field, log_n=rng.randint(8, 22), graph=rng.random() < 0.5)
    if kind == "batch":
        low = rng.randint(10, 14)
        return dict(kind=kind, jobs=rng.randint(3, 80), low=low, high=rng.randint(low + 2, 20),
                    mix=rng.randint(1, 10**6))
    return dict(kind=kind, field=field, n=int(2.0 ** rng.uniform(10, 24)))


# ---------------------------------------------------------------- inputs
def _vector(field, n, gen, device="cuda"):
    """n elements below the modulus, as [n, 8] limbs: seven uniform limbs under
    a top limb uniform below the modulus's own."""
    x = torch.randint(-2**31, 2**31, (n, 8), dtype=torch.int32, device=device, generator=gen)
    top = FIELDS[field][0] >> 224
    x[:, 7] = torch.randint(0, top, (n,), dtype=torch.int32, device=device, generator=gen)
    return x


def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(seed)


def _mont(field, v):
    return (v << 256) % FIELDS[field][0]


def _batch_jobs(case):
    """(field, log_n, inverse) of every job of a batch, from the case alone."""
    rng = random.Random(case["mix"])
    return [(rng.choice(["bls12_381_fr", "bn254_fr"]), rng.randint(case["low"], case["high"]),
             rng.random() < 0.5) for _ in range(case["jobs"])]


def prepare(case, seed):
    gen = _generator(seed)
    kind = case["kind"]
    if kind == "ntt":
        g = _mont(case["field"], FIELDS[case["field"]][1]) if case["coset"] else None
        x = _vector(case["field"], 1 << case["log_n"], gen)
        plan = zk.Plan(case["field"], case["log_n"], inverse=case["inverse"], coset_shift=g,
                       twiddle_mode=case["twiddle"])
        return dict(kind=kind, plan=plan, x=x, out=torch.empty_like(x))
    if kind == "host":
        x = _vector(case["field"], 1 << case["log_n"], gen).cpu().pin_memory()
        plan = zk.Plan(case["field"], case["log_n"], inverse=case["inverse"])
        return dict(kind=kind, plan=plan, x=x, out=torch.empty_like(x).pin_memory())
    if kind == "groth16":
        n = 1 << case["log_n"]
        a, b, c = (_vector(case["field"], n, gen) for _ in range(3))
        s = dict(kind=kind, field=case["field"], log_n=case["log_n"], a=a, b=b, c=c,
                 h=torch.empty_like(a), graph=None,
                 scratch=torch.empty((3 * n, 8), dtype=torch.int32, device="cuda"))
        if case["graph"]:
            torch.cuda.synchronize()
            s["graph"] = zk.Groth16Graph(case["field"], case["log_n"], a, b, c, s["h"],
                                         s["scratch"], torch.cuda.Stream())
        return s
    if kind == "batch":
        plans, kept = [], {}
        for job in _batch_jobs(case):
            if job not in kept:
                kept[job] = zk.Plan(job[0], job[1], inverse=job[2])
            plans.append(kept[job])
        xs = [_vector(f, 1 << log_n, gen) for f, log_n, _ in _batch_jobs(case)]
        # the outputs are places in one buffer, as a server hands out device memory
        arena = torch.empty((sum(len(x) for x in xs), 8), dtype=torch.int32, device="cuda")
        return dict(kind=kind, plans=plans, xs=xs, arena=arena,
                    outs=list(arena.split([len(x) for x in xs])))
    a, b, c = (_vector(case["field"], case["n"], gen) for _ in range(3))
    z = random.Random(seed).randrange(1, FIELDS[case["field"]][0])
    return dict(kind=kind, field=case["field"], a=a, b=b, c=c, z=z, out=torch.empty_like(a))


def run(state):
    kind = state["kind"]
    if kind == "ntt":
        return state["plan"].execute(state["x"], state["out"])
    if kind == "host":
        return state["plan"].execute_host(state["x"], state["out"])
    if kind == "groth16":
        if state["graph"] is not None:
            state["graph"].launch()
            return state["h"]
        return zk.groth16_h(state["field"], state["log_n"], state["a"], state["b"], state["c"],
                            h=state["h"], scratch=state["scratch"])
    if kind == "batch":
        zk.execute_batch(state["plans"], state["xs"], state["outs"])
        return state["arena"]
    return zk.pointwise(state["field"], state["a"], state["b"], state["c"], state["z"],
                        out=state["out"])


# ---------------------------------------------------------------- least work
def _products(log_n):
    """Field products by a twiddle other than 1 in one transform."""
    n = 1 << log_n
    return n // 2 * log_n - (n - 1)


def work(case):
    """Bytes: every input read once, every output written once.  Operations:
    264 32-bit multiply-adds per field product (8 x (8 + 8 + 1) low and high
    halves), the products with a twiddle other than 1 and the scales."""
    kind = case["kind"]
    if kind in ("ntt", "host"):
        n = 1 << case["log_n"]
        scale = n if case["inverse"] or case.get("coset") else 0
        return dict(bytes=64 * n, flops=264 * (_products(case["log_n"]) + scale))
    if kind == "groth16":
        n = 1 << case["log_n"]
        # seven transforms, the three coset scales and three 1/n joined, the
        # last scale, one product of a and b
        return dict(bytes=128 * n, flops=264 * (7 * _products(case["log_n"]) + 5 * n))
    if kind == "batch":
        jobs = _batch_jobs(case)
        return dict(bytes=sum(64 << L for _, L, _ in jobs),
                    flops=264 * sum(_products(L) + ((1 << L) if inv else 0) for _, L, inv in jobs))
    return dict(bytes=128 * case["n"], flops=264 * 2 * case["n"])


# ---------------------------------------------------------------- exact values
def _ints(t):
    b = t.cpu().numpy().view("<u4").tobytes()
    return [int.from_bytes(b[i:i + 32], "little") for i in range(0, len(b), 32)]


def _limbs(v):
    a = np.frombuffer(b"".join(x.to_bytes(32, "little") for x in v), dtype="<i4")
    return torch.from_numpy(a.reshape(-1, 8).copy())


def _transform(v, field, inverse, shift=None):
    """The transform of a list of integers (plain or in Montgomery form: it is
    linear), radix 2 on Python integers."""
    r, g, s = FIELDS[field]
    n = len(v)
    log_n = n.bit_length() - 1
    w = pow(g, (r - 1) >> s, r)
    w = pow(w, 1 << (s - log_n), r)
    if inverse:
        w = pow(w, -1, r)
    if shift is not None and not inverse:
        v, p = list(v), 1
        for i in range(n):
            v[i] = v[i] * p % r
            p = p * shift % r
    out = [v[int(format(i, "0%db" % log_n)[::-1], 2)] for i in range(n)]
    size = 2
    while size <= n:
        half, wl = size // 2, pow(w, n // size, r)
        tw = [1] * half
        for j in range(1, half):
            tw[j] = tw[j - 1] * wl % r
        for lo in range(0, n, size):
            for j in range(half):
                x, y = out[lo + j], out[lo + j + half] * tw[j] % r
                out[lo + j] = (x + y) % r
                out[lo + j + half] = (x - y) % r
        size *= 2
    if inverse:
        p, step = pow(n, -1, r), (1 if shift is None else pow(shift, -1, r))
        for i in range(n):
            out[i] = out[i] * p % r
            p = p * step % r
    return out


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch" or math.log2(case.get("n", 1 << case.get("log_n", 0))) > EXACT_LOG_N:
        return None
    if kind == "groth16" and case["log_n"] > 14:
        return None
    gen = _generator(seed)
    field = case["field"]
    r, g, _ = FIELDS[field]
    if kind in ("ntt", "host"):
        v = _ints(_vector(field, 1 << case["log_n"], gen))
        return _limbs(_transform(v, field, case["inverse"], g if case.get("coset") else None))
    n = case["n"] if kind == "pointwise" else 1 << case["log_n"]
    a, b, c = (_ints(_vector(field, n, gen)) for _ in range(3))
    from_mont = pow(2, -256, r)
    if kind == "pointwise":
        z = random.Random(seed).randrange(1, r)
        return _limbs([(x * y * from_mont - u) * z % r * from_mont % r for x, y, u in zip(a, b, c)])
    a, b, c = (_transform(_transform(v, field, True), field, False, g) for v in (a, b, c))
    z = pow(pow(g, n, r) - 1, -1, r)
    q = [(x * y * from_mont - u) * z % r for x, y, u in zip(a, b, c)]
    return _limbs(_transform(q, field, True, g))
