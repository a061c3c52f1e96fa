"""The workloads this library's speed is judged by: calls that a program using it makes,
with the sizes of the bivariate-bicycle detector models it decodes.

Each case builds its decoding problem (the phenomenological detector matrix of a BB code:
T noisy rounds and one perfect round), samples faults on the GPU from the seed, and calls
one public entry point.  `exact` recomputes the differentiable leg in 64 bits with torch
alone; the decoders return whole numbers only.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

import paper_2511_21660_gb300 as q

# code: (l, m, monomials (power of x, power of y) of A and of B, memory-strength range of
# the legs after the first)
CODES = {
    "bb72": (6, 6, ((3, 0), (0, 1), (0, 2)), ((0, 3), (1, 0), (2, 0)), (-0.24, 0.66)),
    "bb144": (12, 6, ((3, 0), (0, 1), (0, 2)), ((0, 3), (1, 0), (2, 0)), (-0.24, 0.66)),
    "bb288": (12, 12, ((3, 0), (0, 2), (0, 7)), ((0, 3), (1, 0), (2, 0)), (-0.161, 0.815)),
}
MIXED_ROUNDS = (("bb72", 6), ("bb144", 12), ("bb288", 18))   # codes of an uneven batch, mixed 1:2:1
LEGS = 300                                                   # legs after the first


@functools.lru_cache(maxsize=8)
def problem(code, rounds):
    """(M, N, row_ptr, col_idx) of the detector matrix: check (t, i) is row t * m + i; data
    fault (t, q) flips the checks of column q in round t, measurement fault (t, i) flips
    (t, i) and (t + 1, i).  rounds = 0: one fault per qubit (code capacity)."""
    l, m, a, b, _ = CODES[code]
    half = l * m

    def neighbours(i, terms):   # the columns of row i of sum_k x^p y^r
        u, v = divmod(i, m)
        return [((u + p) % l) * m + (v + r) % m for p, r in terms]

    hx = [sorted(neighbours(i, a) + [half + c for c in neighbours(i, b)]) for i in range(half)]
    n, data = 2 * half, (rounds + 1) * 2 * half
    ptr, col = [0], []
    for t in range(rounds + 1):
        for i in range(half):
            row = [t * n + c for c in hx[i]]
            if t > 0:
                row.append(data + (t - 1) * half + i)
            if t < rounds:
                row.append(data + t * half + i)
            col += sorted(row)
            ptr.append(len(col))
    return ((rounds + 1) * half, data + rounds * half, np.array(ptr, dtype=np.int32),
            np.array(col, dtype=np.int32))


@functools.lru_cache(maxsize=8)
def memory_strengths(code, rounds, legs):
    """gamma table [legs + 1, N]: 0.125 in the first leg, uniform draws in the later ones."""
    lo, hi = CODES[code][4]
    N = problem(code, rounds)[1]
    g = np.random.default_rng(7).uniform(lo, hi, (legs + 1, N)).astype(np.float32)
    g[0] = 0.125
    return g


def sample(code, rounds, p, shots, seed):
    """Faults (bool [shots, N]) and syndromes (bool [shots, M]) on the GPU."""
    M, N, ptr, col = problem(code, rounds)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    H = torch.zeros((N, M), dtype=torch.float16, device="cuda")
    rows = np.repeat(np.arange(M), np.diff(ptr))
    H[torch.from_numpy(col.astype(np.int64)).cuda(), torch.from_numpy(rows).cuda()] = 1.0
    F = torch.empty((shots, N), dtype=torch.bool, device="cuda")
    S = torch.empty((shots, M), dtype=torch.bool, device="cuda")
    for s in range(0, shots, 16384):
        e = min(shots, s + 16384)
        F[s:e] = torch.rand((e - s, N), generator=gen, device="cuda") < p
        S[s:e] = (F[s:e].to(torch.float16) @ H).to(torch.int32) & 1   # counts <= 8: exact
    return F, S


def packed(bits):
    """bool [B, n] -> int64 [B, ceil(n / 64)], bit k of word w is entry 64 w + k."""
    B, n = bits.shape
    words = (n + 63) // 64
    out = torch.empty((B, words), dtype=torch.int64, device=bits.device)
    shift = torch.arange(64, dtype=torch.int64, device=bits.device)
    for s in range(0, B, 16384):
        e = min(B, s + 16384)
        wide = torch.zeros((e - s, words * 64), dtype=torch.int64, device=bits.device)
        wide[:, :n] = bits[s:e]
        out[s:e] = (wide.view(e - s, words, 64) << shift).sum(dim=2)
    return out


def decoder(code, rounds, p, legs=LEGS, **options):
    M, N, ptr, col = problem(code, rounds)
    return q.RelayDecoder(ptr, col, np.full(N, p), memory_strengths(code, rounds, legs),
                          q.RelayConfig(legs_after_first=legs, **options))


def listed():
    base = dict(code="bb144", rounds=12, p=0.003, S=5, fp16=False)
    return [
        # one syndrome of the small code: the latency of a single real-time decode
        dict(base, name="decode_bb72_1", kind="decode", code="bb72", rounds=6, shots=1),
        # code-capacity shots of a threshold study: tiny graphs, many of them
        dict(base, name="decode_bb72_capacity", kind="decode", code="bb72", rounds=0, p=0.05,
             shots=65536),
        # the codes of a small processor, one window each: fewer shots than SMs
        dict(base, name="decode_gross_100", kind="decode", shots=100),
        # the headline workload: a Monte-Carlo batch of the gross code
        dict(base, name="decode_gross_100k", kind="decode", shots=100000),
        # the same with binary16 message storage, an odd batch
        dict(base, name="decode_gross_fp16", kind="decode", shots=20011, fp16=True),
        # the largest graph of the configurations (two-gross code, 18 rounds)
        dict(base, name="decode_two_gross", kind="decode", code="bb288", rounds=18, shots=16384),
        # high noise: some shots never converge and run every leg
        dict(base, name="decode_gross_hard", kind="decode", p=0.02, shots=10007),
        # a host program: numpy buffers in and out, first solution only
        dict(base, name="host_gross_first", kind="host", S=1, shots=50021),
        # shots of three codes in one call
        dict(base, name="grouped_codes", kind="grouped", shots=32768),
        # first leg, then filtered-OSD / the cluster decoder on what it leaves
        dict(base, name="leg_then_osd", kind="osd", p=0.02, shots=50000),
        dict(base, name="leg_then_cluster", kind="cluster", p=0.02, shots=50000),
        # one gradient step of the memory-strength tuning
        dict(base, name="soft_step", kind="soft", p=0.02, shots=2048, iterations=25, every=5,
             fp64=False),
    ]


def draw(rng):
    kind = rng.choice(["decode", "decode", "decode", "hard", "host", "grouped", "mixed", "osd",
                       "cluster", "soft"])
    log = lambda lo, hi: int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))  # noqa: E731
    case = dict(kind=kind, code="bb144", rounds=rng.randint(7, 13),
                p=round(rng.uniform(0.001, 0.004), 5), S=rng.choice([1, 3, 5]),
                fp16=rng.random() < 0.25)
    if kind == "decode":
        case["code"] = rng.choice(["bb72", "bb144", "bb144", "bb288"])
        case["rounds"] = {"bb72": rng.choice([0, rng.randint(4, 7)]), "bb144": rng.randint(8, 13),
                          "bb288": rng.randint(12, 18)}[case["code"]]
        if case["rounds"] == 0:
            case["p"] = 0.05
        case["shots"] = log(1, {"bb72": 100000, "bb144": 60000, "bb288": 16000}[case["code"]])
    elif kind == "hard":
        case.update(kind="decode", p=0.02, shots=log(500, 8000), fp16=False,
                    rounds=rng.randint(11, 12))
    elif kind == "host":
        case["shots"] = log(1, 50000)
    elif kind in ("grouped", "mixed"):
        case.update(rounds=12, shots=log(300, 30000))
    elif kind in ("osd", "cluster"):
        case.update(rounds=rng.randint(10, 12), p=0.02, S=1, fp16=False, shots=log(2000, 40000))
    else:
        fp64 = rng.random() < 0.3
        every = rng.choice([1, 3, 5])
        case.update(code="bb72" if fp64 else "bb144", p=0.02, S=1, fp16=False,
                    rounds=rng.randint(4, 6) if fp64 else rng.randint(8, 12), fp64=fp64,
                    iterations=rng.randint(8, 25), every=every,
                    shots=log(32, 256) if fp64 else log(100, 2000))
    return case


class State:
    pass


def prepare(case, seed):
    s = State()
    s.case, kind = case, case["kind"]
    code, rounds, p, shots = case["code"], case["rounds"], case["p"], case["shots"]
    opts = dict(stop_after_solutions=case["S"],
                msg_precision=q.QLDPC_MSG_FP16 if case["fp16"] else q.QLDPC_MSG_FP32)
    if kind in ("grouped", "mixed"):
        gen = torch.Generator(device="cuda")
        gen.manual_seed(seed)
        kinds = torch.tensor([0, 1, 1, 2], dtype=torch.int32, device="cuda")
        s.codes = kinds[torch.randint(0, 4, (shots,), generator=gen, device="cuda")].contiguous()
        s.decs = [decoder(c, r, p, **opts) for c, r in MIXED_ROUNDS]
        s.syn = torch.zeros((shots, max(d.syndrome_words for d in s.decs)), dtype=torch.int64,
                            device="cuda")
        for k, (c, r) in enumerate(MIXED_ROUNDS):
            here = torch.nonzero(s.codes == k).flatten()
            if here.numel():
                w = packed(sample(c, r, p, here.numel(), 3 * seed + k)[1])
                s.syn[here, :w.shape[1]] = w
        return s
    F, S = sample(code, rounds, p, shots, seed)
    s.syn = packed(S)
    M, N, ptr, col = problem(code, rounds)
    if kind == "soft":
        real = torch.float64 if case["fp64"] else torch.float32
        s.faults = packed(F)
        s.gamma, s.alpha = (t.to(real).requires_grad_() for t in strengths(N, case, seed))
        s.soft = q.SoftDMem(ptr, col, np.full(N, p), iterations=case["iterations"],
                            checkpoint_every=case["every"], dtype=real)
        return s
    if kind in ("osd", "cluster"):
        s.first = decoder(code, rounds, p, legs=0)
        prior = np.full(N, p)
        s.post = (q.FilteredOSD(ptr, col, prior, 25, 8.0, 500) if kind == "osd" else
                  q.ClusterDecoder(ptr, col, prior, 25, -0.5, 4.5, 128, 512))
        return s
    s.dec = decoder(code, rounds, p, **opts)
    if kind == "host":
        pin = lambda *shape, dt: torch.empty(shape, dtype=dt, pin_memory=True).numpy()  # noqa: E731
        s.syn = s.syn.cpu().pin_memory().numpy().view(np.uint64)
        s.out = (pin(shots, s.dec.correction_words, dt=torch.int64).view(np.uint64),
                 pin(shots, dt=torch.int32), pin(shots, dt=torch.uint8),
                 pin(shots, dt=torch.int32))
    return s


def strengths(N, case, seed):
    """gamma [N] and alpha [T] in the middle of a tuning run (float32 values)."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed + 1000003)
    g = 0.05 + 0.15 * torch.rand(N, generator=gen, device="cuda")
    a = 0.3 + 0.2 * torch.rand(case["iterations"], generator=gen, device="cuda")
    return g, a


def run(s):
    kind = s.case["kind"]
    if kind == "decode":
        return s.dec.decode(s.syn)
    if kind == "host":
        return s.dec.decode_host(s.syn, out=s.out)
    if kind == "grouped":
        return q.decode_grouped(s.decs, s.codes, s.syn)
    if kind == "mixed":
        return q.decode_mixed(s.decs, s.codes, s.syn)
    if kind == "osd":
        return q.first_leg_then_osd(s.first, s.post, s.syn)
    if kind == "cluster":
        return q.first_leg_then_cluster(s.first, s.post, s.syn)
    loss = q.soft_dmem_loss(s.soft, s.syn, s.faults, s.gamma, s.alpha)
    return (loss.detach(), *torch.autograd.grad(loss, (s.gamma, s.alpha)))


def work(case):
    """Bytes: packed syndromes in, packed corrections and the per-shot numbers out.  Operations:
    13 per edge and decoding iteration (check rule 7, fault rule 5, decision 1); the
    differentiable leg takes about 30 per edge and iteration, forward and backward together.
    Iterations per shot: at low noise one per solution and 0.6 more in the first leg; at
    p = 0.02 the mean of full Relay over many shots, or of its first leg alone; for the
    code-capacity shots at p = 0.05 their mean with five solutions."""
    kind, shots = case["kind"], case["shots"]
    if kind in ("grouped", "mixed"):
        parts = [(problem(c, r), f) for (c, r), f in zip(MIXED_ROUNDS, (0.25, 0.5, 0.25))]
    else:
        parts = [(problem(case["code"], case["rounds"]), 1.0)]
    total = {"bytes": 0.0, "flops": 0.0}
    for (M, N, ptr, col), share in parts:
        words = (M + 63) // 64 + (N + 63) // 64
        E, n = len(col), shots * share
        if kind == "soft":
            real = 8 if case["fp64"] else 4
            total["bytes"] += 8 * words * n + real * (2 * N + 2 * case["iterations"] + 1)
            total["flops"] += 30.0 * E * case["iterations"] * n
            continue
        if kind not in ("grouped", "mixed") and case["rounds"] == 0:
            iters = 11.9
        elif case["p"] >= 0.02:
            iters = 10.2 if kind in ("osd", "cluster") else 43.6
        else:
            iters = case["S"] + 0.6
        total["bytes"] += (8 * words + 9) * n
        total["flops"] += 13.0 * E * iters * n
    return total


def exact(case, seed):
    """The differentiable leg in 64 bits: sum-product messages with memory terms, the binary
    cross-entropy of the marginals against the sampled faults, and its gradients."""
    if case["kind"] != "soft":
        return None
    M, N, ptr, col = problem(case["code"], case["rounds"])
    F, S = sample(case["code"], case["rounds"], case["p"], case["shots"], seed)
    g, a = (t.double().requires_grad_() for t in strengths(N, case, seed))
    eps = 1e-15 if case["fp64"] else 2.0 ** -23
    w = math.log((1.0 - case["p"]) / case["p"])
    if not case["fp64"]:
        w = float(np.float32(w))
    deg = np.diff(ptr)
    D = int(deg.max())
    # edges as [M, D] with padding slots that take column N (a column of infinite belief)
    cols = np.full((M, D), N, dtype=np.int64)
    for i in range(M):
        cols[i, :deg[i]] = col[ptr[i]:ptr[i + 1]]
    real = torch.from_numpy(cols < N).cuda()
    flat = torch.from_numpy(cols.reshape(-1)).cuda()
    loss_sum, gg, ga = 0.0, torch.zeros_like(g), torch.zeros_like(a)
    for s in range(0, case["shots"], 128):
        f = F[s:s + 128].double()
        sign = torch.where(S[s:s + 128], -1.0, 1.0).double()[:, :, None]
        b = f.shape[0]
        L = torch.full((b, N), w, dtype=torch.float64, device="cuda")
        nu = torch.full((b, M, D), w, dtype=torch.float64, device="cuda")
        for t in range(case["iterations"]):
            lam = (1.0 - g) * w + g * L
            tau = torch.where(real, torch.tanh(nu / 2), torch.ones((), dtype=torch.float64,
                                                                   device="cuda"))
            one = torch.ones((b, M, 1), dtype=torch.float64, device="cuda")
            left = torch.cumprod(torch.cat([one, tau[:, :, :-1]], 2), 2)
            right = torch.cumprod(torch.cat([one, tau.flip(2)[:, :, :-1]], 2), 2).flip(2)
            P = torch.clamp(left * right, -(1.0 - eps), 1.0 - eps)
            mu = torch.where(real, a[t] * sign * 2.0 * torch.atanh(P), 0.0)
            into = torch.zeros((b, N + 1), dtype=torch.float64, device="cuda")
            into = into.index_add(1, flat, mu.reshape(b, -1))
            L = lam + into[:, :N]
            nu = torch.cat([L, L[:, :1]], 1)[:, flat].reshape(b, M, D) - mu
        sp = torch.nn.functional.softplus
        loss = (f * sp(L, threshold=700) + (1.0 - f) * sp(-L, threshold=700)).sum()
        x, y = torch.autograd.grad(loss, (g, a))
        loss_sum, gg, ga = loss_sum + loss.detach(), gg + x, ga + y
    scale = 1.0 / (case["shots"] * N)
    return loss_sum * scale, gg * scale, ga * scale
