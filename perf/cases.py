"""The calls whose time counts: what a user of the framework has it do, through its public entry points.

Sizes are the ones of the repository's own workloads (inputs.CONFIG_SIZES, bench.py, the tests) or plain fractions of
them; `draw` spreads the same calls over their whole ranges.  The int32 and int8 tensor forms and the staged engine
are comparators of the default path and are not listed.
"""
import math

import numpy as np
import torch

from paper_2502_12428_gb300 import inputs
import paper_2502_12428_gb300.qfs as qfs

# Share of quartics past the height-1 test and theta steps per such quartic, as the repository's own workloads have
# them (they only weigh the operation counts of `work`).
PAST_HEIGHT_1 = {"dense": {3: 0.37, 5: 0.21, 7: 0.145, 11: 0.091, 13: 0.077}, "sparse": 0.38}
THETA_STEPS = {"dense": 1.25, "sparse": 4.4}


def listed():
    return [
        # The smallest call: 64 quartics and the Fermat quartic over F_3.  Launches and latency.
        dict(name="heights_p3_65", op="heights", p=3, n=65, kind="dense", power="chain"),
        # One step of a search that hands over a thousand candidates at a time, an odd count: about 145 of them pass
        # the height-1 test, fewer than the GPU could hold at once.
        dict(name="heights_p7_1001", op="heights", p=7, n=1001, kind="dense", power="chain"),
        # The p = 5 workload: random quartics, the default mode.
        dict(name="heights_p5_65536", op="heights", p=5, n=65536, kind="dense", power="chain"),
        # Sparse quartics at p = 5: zero taps, many quartics past height 1, uneven numbers of theta steps.
        dict(name="heights_p5_sparse_131071", op="heights", p=5, n=131071, kind="sparse", power="chain"),
        # The headline workload, and the largest call: p = 7, random quartics, the default mode.
        dict(name="heights_p7_262144", op="heights", p=7, n=262144, kind="dense", power="chain"),
        # Three primes in one launch, every quartic beside its image under a change of variables (the invariance
        # check a user runs); p = 11 brings the largest forms.
        dict(name="heights_mixed", op="mixed", n5=8192, n7=8192, n11=256),
        # The identity power mode: the same Delta_1 array without the chain.
        dict(name="heights_p7_identity_65536", op="heights", p=7, n=65536, kind="dense", power="identity"),
        # The reduced power mode: a search over as many quartics as possible.
        dict(name="heights_p7_reduced_262144", op="heights", p=7, n=262144, kind="dense", power="reduced"),
        # Export of the theta matrices of a few quartics (8.6 MB each at p = 7).
        dict(name="theta_matrix_p7_48", op="theta_matrix", p=7, n=48),
        # The mod-p matrix product at the paper's smallest size.
        dict(name="matmul_mod11_5000", op="matmul", p=11, n=5000, m=5000, k=5000),
        # Exact powering over Z of a degree-16 form: the smallest and the largest exponent of the paper's workload.
        dict(name="poly_power_d16_n5", op="poly_power", d=16, n=5),
        dict(name="poly_power_d16_n15", op="poly_power", d=16, n=15),
    ]


def _log_int(rng, lo, hi):
    """An integer in [lo, hi], uniform in its logarithm."""
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    op = rng.choice(["heights", "heights", "heights", "mixed", "theta_matrix", "matmul", "poly_power"])
    if op == "heights":
        power = rng.choice(["chain", "chain", "chain", "identity", "reduced"])
        p = rng.choice([3, 5, 5, 7, 7, 11] + [13] * (power == "reduced"))
        kind = rng.choice(["dense", "dense", "sparse"])
        top = {"chain": {3: 262144, 5: 131072, 7: 65536, 11: 256}, "identity": {3: 262144, 5: 262144, 7: 65536, 11: 512},
               "reduced": {3: 262144, 5: 262144, 7: 262144, 11: 16384, 13: 2048}}[power][p]
        return dict(op="heights", p=p, n=_log_int(rng, 33, top), kind=kind, power=power)
    if op == "mixed":
        return dict(op="mixed", n5=_log_int(rng, 64, 8192), n7=_log_int(rng, 64, 8192), n11=_log_int(rng, 8, 256))
    if op == "theta_matrix":
        p = rng.choice([3, 5, 7])
        return dict(op="theta_matrix", p=p, n=_log_int(rng, 1, {3: 4096, 5: 512, 7: 64}[p]))
    if op == "matmul":
        return dict(op="matmul", p=rng.choice([2, 7, 11, 11, 13, 31, 101, 251, 256]), n=_log_int(rng, 64, 5000),
                    m=_log_int(rng, 64, 5000), k=_log_int(rng, 64, 5000))
    d = rng.choice([4, 8, 16, 16])
    return dict(op="poly_power", d=d, n=rng.randint(2, {4: 40, 8: 24, 16: 15}[d]))


def _quartics(p, n, kind, seed):
    """n rows of 35 coefficients (host); dense batches end with the Fermat quartic."""
    if kind == "sparse":
        return inputs.sparse(p, n, seed)
    f = inputs.dense(p, n, seed)
    f[-1] = inputs.fermat()
    return f


def _device(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def prepare(case, seed):
    seed = (0x5EED0000 + 7919 * int(seed)) & 0x7FFFFFFFFFFF
    op = case["op"]
    if op == "heights":
        return dict(case, f=_device(_quartics(case["p"], case["n"], case["kind"], seed)))
    if op == "mixed":
        groups = []
        for p, n in ((5, case["n5"]), (7, case["n7"]), (11, case["n11"])):
            f = inputs.dense(p, n, seed + p)
            image = inputs.substitute(f, inputs.pgl4_matrices(p, n, seed + 100 + p), p)
            groups.append((p, _device(np.concatenate([f, image])), None))
        return dict(case, groups=groups)
    if op == "theta_matrix":
        return dict(case, f=_device(inputs.dense(case["p"], case["n"], seed)))
    if op == "matmul":
        g = torch.Generator(device="cuda").manual_seed(seed)
        A = torch.randint(0, case["p"], (case["n"], case["k"]), dtype=torch.uint8, device="cuda", generator=g)
        B = torch.randint(0, case["p"], (case["k"], case["m"]), dtype=torch.uint8, device="cuda", generator=g)
        return dict(case, A=A, B=B)
    # a form with coefficients in {0..4}, as host integers
    rng = np.random.default_rng(seed)
    return dict(case, c=rng.integers(0, 5, math.comb(case["d"] + 3, 3), dtype=np.uint32))


def run(state):
    op = state["op"]
    if op == "heights":
        return qfs.heights(state["p"], state["f"], power=state["power"])
    if op == "mixed":
        return qfs.heights_multi(state["groups"])
    if op == "theta_matrix":
        return qfs.theta_matrix(state["p"], state["f"])
    if op == "matmul":
        return qfs.matmul_mod(state["p"], state["A"], state["B"])
    return qfs.poly_power_limbs(state["d"], state["c"], state["n"])


def _forms(d):
    return math.comb(d + 3, 3)


def _theta_terms(p):
    """Nonzero entries of the theta matrix: the pairs r, c of degree-4(p-1) monomials with every exponent of
    p r + (p-1)1 - c at least 0 and their sum right, that is c <= p r + (p-1)1 exponent by exponent."""
    d = 4 * (p - 1)
    total = 0
    # c = p c' + rho with rho in [0, p)^4: c' <= r, so each residue class of kernel degree k has C(k+3,3) C(d-k+3,3)
    count = [0] * (d + 1)
    count[0] = 1
    for _ in range(4):
        count = [sum(count[s - r] for r in range(p) if s >= r) for s in range(d + 1)]
    for k in range(4):
        total += count[d - p * k] * _forms(k) * _forms(d - k) if d - p * k >= 0 else 0
    return total


def _height_macs(p, n, kind, power):
    """Multiply-adds of the named power mode over n quartics, with the expected share past height 1."""
    past = PAST_HEIGHT_1["sparse"] if kind == "sparse" else PAST_HEIGHT_1["dense"][p]
    steps = THETA_STEPS[kind]
    fedder = sum(_forms(4 * k) * 35 for k in range(1, (p - 1) // 2)) + _forms(2 * (p - 1))
    to_g = sum(_forms(4 * k) * 35 for k in range(1, p - 1))
    if power == "chain":
        later = sum(_forms(4 * k) * 35 for k in range(p - 1, p * (p - 1))) + steps * _theta_terms(p)
    elif power == "identity":
        dm, d1 = 4 * (p - 2), 4 * p
        later = 35 * _forms(4 * (p - 1)) + to_g + _forms(dm) * _forms(d1) + steps * _theta_terms(p)
    else:
        # theta(F) = -f^(p-2) u(F Delta_1(f)): 35 outputs of u, then a 35-tap product
        later = 35 * _forms(4 * (p - 1)) + steps * (35 * _forms(4 * (p - 1)) + 35 * _forms(4 * (p - 2)))
    return n * (fedder + past * (to_g + later))


def work(case):
    op = case["op"]
    if op == "heights":
        return {"bytes": 36 * case["n"], "flops": int(2 * _height_macs(case["p"], case["n"], case["kind"], case["power"]))}
    if op == "mixed":
        groups = ((5, case["n5"]), (7, case["n7"]), (11, case["n11"]))
        return {"bytes": 72 * sum(n for _, n in groups),
                "flops": int(4 * sum(_height_macs(p, n, "dense", "chain") for p, n in groups))}
    if op == "theta_matrix":
        p, n = case["p"], case["n"]
        ld = _forms(4 * (p - 1))
        chain = sum(_forms(4 * k) * 35 for k in range(1, p * (p - 1)))
        return {"bytes": n * (35 + ld * ld), "flops": 2 * n * chain}
    if op == "matmul":
        n, m, k = case["n"], case["m"], case["k"]
        return {"bytes": n * k + k * m + n * m, "flops": 2 * n * m * k}
    # products of residues: a transform of the output's length each way for every 31 bits of a coefficient
    d, n = case["d"], case["n"]
    length = (d * n + 1) ** 3
    words = max(1, math.ceil(n * math.log2(2 * _forms(d) + 1) / 31))
    return {"bytes": 4 * _forms(d) + 32 * _forms(d * n), "flops": int(2 * words * length * math.log2(length))}


def _product(a, b, mod):
    """Product of two batches of polynomials in (e2, e3, e4), arrays (n, S, S, S), reduced mod `mod`."""
    S, T = a.shape[1], b.shape[1]
    out = np.zeros((a.shape[0],) + (S + T - 1,) * 3, np.int64)
    for i, j, k in np.argwhere(b.any(axis=0)):
        out[:, i:i + S, j:j + S, k:k + S] += a * b[:, i, j, k][:, None, None, None]
    return out % mod


def _exact_heights_p3(f):
    """Heights over F_3 by the definition: Fedder's test on g = f^2, Delta = (lift(g)^3 - sum of cubed terms) / 3,
    then g <- u(Delta g) until the coefficient of (x1 x2 x3 x4)^2 is nonzero, the iterate is zero or h = 10."""
    p, n = 3, f.shape[0]
    F = np.zeros((n, 5, 5, 5), np.int64)
    for i, (_, e2, e3, e4) in enumerate(inputs.MONOMIALS):
        F[:, e2, e3, e4] = f[:, i]
    g = _product(F, F, p)
    cube = _product(_product(g, g, p * p), g, p * p)
    cube[:, ::3, ::3, ::3] -= g ** 3
    delta = cube % (p * p) // p
    D, d = 24, 8
    room = np.zeros((n, 3 * d + 3 + d, 3 * d + 3 + d, 3 * d + 3 + d), np.int64)   # index e + d, zeros around
    room[:, d:d + D + 1, d:d + D + 1, d:d + D + 1] = delta
    e = np.arange(d + 1)
    inside = (e[:, None, None] + e[None, :, None] + e[None, None, :]) <= d
    h = np.where(g[:, 2, 2, 2] != 0, 1, 0)
    live = h == 0
    for step in range(2, 11):
        out = np.zeros_like(g)
        for a, b, c in np.argwhere(inside):
            s = [slice(p - 1 - x + d, p - 1 - x + d + p * d + 1, p) for x in (a, b, c)]
            out += g[:, a, b, c][:, None, None, None] * room[:, s[0], s[1], s[2]]
        # the exponent of x1 of p r + (p-1)1 - c is that of degree 24 and is checked by Delta's own zeros
        g = np.where(inside, out % p, 0)
        hit = live & (g[:, 2, 2, 2] != 0)
        h[hit] = step
        live &= ~hit & g.any(axis=(1, 2, 3))
    return h


def exact(case, seed):
    if case["op"] == "heights" and case["p"] == 3 and case["n"] <= 256:
        s = prepare(case, seed)
        return torch.from_numpy(_exact_heights_p3(s["f"].cpu().numpy().astype(np.int64)).astype(np.int8))
    if case["op"] == "matmul":
        # products of residues below 256 over at most 5,000 terms stay below 2^53
        s = prepare(case, seed)
        return (s["A"].double() @ s["B"].double()).remainder_(case["p"]).to(torch.uint8)
    return None
