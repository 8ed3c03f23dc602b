"""Performance cases: the work that a user of the decoder has it do, one pass
of each through the public entry points of ``paper_2605_14170_gb300.mbbp``.

The framework decodes batches of syndromes on R redundant representations of
a CSS check matrix, produces and judges Monte-Carlo shots, and trains weighted
min-sum (WMS) weights.  The listed cases take the codes, representation
counts, iteration limits and error rates of its benchmark and tests, from one
shot (a decoder in a control loop) to batches that fill the GPU many times
over; ``draw`` gives more cases of the same kinds with other codes, batches,
error rates and options.

A case is a dict of plain values:
  kind    "decode" (a batch of syndromes), "realtime" (a few shots through the
          entry point that needs no workspace), "montecarlo" (sample, syndrome,
          decode, judge, both error types), "mixed" (several codes at once),
          "train" (WMS loss and gradients), "wms_decode" (learned weights)
  code    "bb72", "bb144", "bb288", "gb882" or "gb" (a generalized bicycle
          code of length 2 L from two seeded polynomials of `weight` terms)
  R, batch, p (error rate of the decoded type), iters, alpha and options.
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

from paper_2605_14170_gb300 import mbbp
from paper_2605_14170_gb300.inputs import gb_code, named_code

BASES_SEED = 20260514   # root orders of the representations: a program keeps them
LMAX = 1.0e4            # the min of the check rule also runs over this value

# (representations, iteration limit) of the mixed case's codes
MIXED = (("bb72", 8), ("bb144", 16), ("bb288", 32))


def listed():
    return [
        # a decoder inside a control loop: one syndrome, latency is all
        dict(name="realtime_bb72_one_shot", kind="realtime", code="bb72", R=4, batch=1, p=0.05, iters=50, alpha=0.625),
        # the [[72,12,6]] configuration: a short batch, launch-bound
        dict(name="decode_bb72_2000", kind="decode", code="bb72", R=4, batch=2000, p=0.05, iters=50, alpha=0.625),
        # a Monte-Carlo step of the batched [[144,12,12]] configuration at a
        # moderate depolarizing rate, with everything around the decoder
        dict(name="montecarlo_bb144", kind="montecarlo", code="bb144", R=16, batch=200_000, p=0.04, iters=100,
             alpha=0.625),
        # the same configuration's noisiest point (depolarizing 0.08: marginal
        # 0.0533), one error type: most of that benchmark's time
        dict(name="decode_bb144_noisy", kind="decode", code="bb144", R=16, batch=200_000, p=0.0533, iters=100,
             alpha=0.625),
        # a longer code with many representations, odd batch
        dict(name="decode_bb288_r32", kind="decode", code="bb288", R=32, batch=20_011, p=0.04, iters=100, alpha=0.625),
        # the length-882 code with the most representations a handle takes
        dict(name="decode_gb882_r64", kind="decode", code="gb882", R=64, batch=5_000, p=0.0333, iters=100, alpha=0.625),
        # the published setting: serial schedule, alpha 0.875, least-metric
        # selection, independent X errors
        dict(name="serial_bb288_lms", kind="decode", code="bb288", R=20, batch=20_000, p=0.06, iters=100, alpha=0.875,
             schedule="serial", decision="lms"),
        # the other check rule
        dict(name="sumproduct_bb144", kind="decode", code="bb144", R=16, batch=4_000, p=0.04, iters=100, alpha=0.625,
             rule="sp"),
        # rows of weight 8, an LLR vector per shot (soft information), ragged
        # sizes
        dict(name="soft_gb254_weight8", kind="decode", code="gb", L=127, weight=4, code_seed=127, R=8, batch=3_001,
             p=0.04, iters=60, alpha=0.75, soft=True),
        # one training step of the weights: forward, loss, adjoint
        dict(name="train_bb144", kind="train", code="bb144", R=8, batch=4_096, p=0.04, T=25, ckpt=5),
        # decoding with learned weights on the length-882 code
        dict(name="wms_decode_gb882", kind="wms_decode", code="gb882", R=64, batch=2_000, p=0.0333, iters=100, T=25),
        # three codes, both error types, in one persistent batch
        dict(name="mixed_three_codes", kind="mixed", batch=10_000, p=0.0333, iters=100, alpha=0.625),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw_code(rng, small=False):
    """A code of the configurations, or a seeded generalized bicycle code."""
    name = rng.choice(["bb72", "bb144", "bb288", "gb"] + ([] if small else ["gb882", "gb"]))
    if name != "gb":
        return dict(code=name)
    weight = rng.choice([3, 3, 3, 4, 5])
    return dict(code="gb", L=rng.randint(24, 96 if small else 240), weight=weight, code_seed=rng.randint(0, 10**6))


def _draw(rng):
    kind = rng.choice(["decode"] * 5 + ["realtime", "montecarlo", "train", "wms_decode", "mixed"])
    p = round(rng.uniform(0.01, 0.055), 4)
    if kind == "mixed":
        return dict(kind=kind, batch=_log(rng, 50, 10_000), p=p, iters=rng.choice([50, 100]), alpha=0.625)
    c = dict(kind=kind, **_draw_code(rng, small=kind == "train"))
    c["R"] = rng.choice([1, 4, 8, 16, 20]) if c["code"] != "gb882" else rng.choice([16, 64])
    c["p"] = p
    if kind == "realtime":
        c.update(batch=_log(rng, 1, 64), iters=rng.choice([30, 50, 100]), alpha=rng.choice([0.625, 0.75]))
    elif kind == "montecarlo":
        c.update(batch=_log(rng, 200, 200_000), iters=100, alpha=0.625)
    elif kind == "train":
        T = rng.randint(5, 25)
        c.update(R=rng.choice([2, 4, 8]), batch=_log(rng, 64, 4_096), T=T, ckpt=rng.randint(1, T))
    elif kind == "wms_decode":
        c.update(batch=_log(rng, 32, 20_000), iters=rng.choice([25, 50, 100]), T=rng.randint(5, 25))
    else:
        c.update(batch=_log(rng, 16, 200_000), iters=rng.choice([20, 50, 100]),
                 alpha=rng.choice([0.625, 0.75, 0.875]))
        if rng.random() < 0.3:
            c["schedule"] = "serial"
        if rng.random() < 0.25:
            c["decision"] = "lms"
        if rng.random() < 0.2:
            c["rule"] = "sp"
        if rng.random() < 0.25:
            c["soft"] = True
    return c


def draw(rng: random.Random):
    c = _draw(rng)
    limit = max(work(x)["flops"] for x in listed())
    while work(c)["flops"] > limit:
        c["batch"] = max(1, int(c["batch"] * 0.6))
    return c


# --------------------------------------------------------------------- inputs

def _code(case):
    name = case["code"]
    if name == "gb882":  # the seeded length-882 generalized bicycle code
        return gb_code(441, [54, 112, 218], [142, 225, 374])
    if name == "gb":
        L, weight = case["L"], case["weight"]
        rng = random.Random(case["code_seed"])
        a, b = (sorted(rng.sample(range(L), weight)) for _ in range(2))
        return gb_code(L, a, b)
    return named_code(name)


def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _errors(g, batch, n, p):
    return torch.rand((batch, n), generator=g, device="cuda") < p


def _syndromes(e, H):
    """H e over GF(2), uint8 [batch, m]."""
    Ht = torch.from_numpy(np.ascontiguousarray(H.T)).to("cuda", torch.float32)
    return (e.to(torch.float32) @ Ht).to(torch.int32).bitwise_and_(1).to(torch.uint8)


def _llr(n, p):
    return torch.full((n,), math.log((1.0 - p) / p), dtype=torch.float32, device="cuda")


def _pack(bits):
    """bool [batch, n] -> int32 words [batch, ceil(n / 32)], bit i of word w =
    entry 32 w + i."""
    batch, n = bits.shape
    W = (n + 31) // 32
    x = torch.zeros((batch, W * 32), dtype=torch.int64, device=bits.device)
    x[:, :n] = bits
    words = (x.view(batch, W, 32) << torch.arange(32, device=bits.device)).sum(-1)
    return torch.where(words >= 2**31, words - 2**32, words).to(torch.int32)


def _outputs(B, batch):
    def new(shape, dtype):
        return torch.empty(shape, dtype=dtype, device="cuda")
    return dict(e_hat=new((batch, B.n), torch.uint8), conv=new((batch, B.R), torch.uint8),
                success=new((batch,), torch.uint8), iters_run=new((batch, B.R), torch.int16),
                selected=new((batch,), torch.int16))


def _workspace(nbytes):
    return torch.empty(nbytes, dtype=torch.uint8, device="cuda")


def _weights(g, R, T, E):
    """Weights and damping as training leaves them: around the normalization
    constant, damping small and often zero."""
    w = 0.625 + 0.1 * torch.randn((R, T, E), generator=g, device="cuda")
    d = 0.1 * torch.randn((R, T, E), generator=g, device="cuda")
    return w.clamp_(0.0, 2.0), d.clamp_(0.0, 0.9)


def prepare(case, seed):
    kind, g = case["kind"], _generator(seed)
    st = {"case": case}
    if kind == "mixed":
        Bs, synd, llrs = [], [], []
        for name, R in MIXED:
            code = named_code(name)
            for H in (code.HZ, code.HX):
                Bs.append(mbbp.mbbp_build_bases(H, R, BASES_SEED))
                synd.append(_syndromes(_errors(g, case["batch"], code.n, case["p"]), H))
                llrs.append(_llr(code.n, case["p"]))
        st["plan"] = mbbp.mbbp_plan_create(Bs)
        st["ios"], st["ws"] = mbbp.mixed_buffers(st["plan"], synd, llrs)
        return st
    code, batch = _code(case), case["batch"]
    n = code.n
    if kind == "montecarlo":
        st["seed"], st["W"], st["n"] = seed, (n + 31) // 32, n
        st["types"] = []
        for H, Ho in ((code.HZ, code.HX), (code.HX, code.HZ)):
            B = mbbp.mbbp_build_bases(H, case["R"], BASES_SEED)
            st["types"].append(dict(B=B, L=mbbp.mbbp_logicals_build(H, Ho), out=_outputs(B, batch),
                                    e=torch.empty((batch, st["W"]), dtype=torch.int32, device="cuda"),
                                    s=torch.empty((batch, B.m), dtype=torch.uint8, device="cuda"),
                                    fail=torch.empty((batch,), dtype=torch.uint8, device="cuda"),
                                    counts=torch.zeros(3, dtype=torch.int64, device="cuda")))
        st["llr"] = _llr(n, 2.0 * case["p"] / 3.0)
        st["ws"] = _workspace(max(mbbp.mbbp_decode_workspace_size(x["B"], batch) for x in st["types"]))
        return st
    B = st["B"] = mbbp.mbbp_build_bases(code.HZ, case["R"], BASES_SEED)
    e = _errors(g, batch, n, case["p"])
    st["s"] = _syndromes(e, code.HZ)
    if case.get("soft"):
        # reliabilities per qubit and shot: the channel's LLR scaled by what a
        # soft measurement adds, lower where an error happened
        x = _llr(n, case["p"]) * (0.5 + torch.rand((batch, n), generator=g, device="cuda"))
        st["llr"] = torch.where(e, 0.5 * x, x).contiguous()
    else:
        st["llr"] = _llr(n, case["p"])
    if kind == "train":
        T, E = case["T"], int(B.edges.max())
        st["w"], st["g"] = _weights(g, B.R, T, E)
        st["gw"], st["gg"] = torch.empty_like(st["w"]), torch.empty_like(st["g"])
        st["etrue"] = _pack(e)
        st["post"] = torch.empty((batch, B.R, n), dtype=torch.float32, device="cuda")
        st["loss"] = torch.empty((batch, B.R), dtype=torch.float32, device="cuda")
        st["ws"] = _workspace(mbbp.mbbp_wms_workspace_size(B, batch, T, case["ckpt"]))
        return st
    st["out"] = _outputs(B, batch)
    if kind == "wms_decode":
        st["w"], st["g"] = _weights(g, B.R, case["T"], int(B.edges.max()))
        st["ws"] = _workspace(mbbp.mbbp_wms_decode_workspace_size(B, batch, case["T"]))
    elif kind == "decode":
        st["ws"] = _workspace(mbbp.mbbp_decode_workspace_size(B, batch))
        st["opt"] = mbbp.Options(
            mbbp.RULE_SP if case.get("rule") == "sp" else mbbp.RULE_NMS, case["alpha"],
            mbbp.SCHEDULE_SERIAL if case.get("schedule") == "serial" else mbbp.SCHEDULE_FLOODING,
            mbbp.DECISION_LMS if case.get("decision") == "lms" else mbbp.DECISION_FWS)
    return st


# ----------------------------------------------------------------- one pass

def _decode_outputs(out):
    return [out["e_hat"], out["conv"], out["success"], out["iters_run"], out["selected"]]


def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind == "mixed":
        mbbp.mbbp_decode_mixed(st["plan"], st["ios"], case["iters"], case["alpha"], mbbp.RULE_NMS, st["ws"])
        return [[x["e_hat"], x["conv"], x["success"], x["iters"], x["selected"]] for x in st["ios"]]
    if kind == "montecarlo":
        X, Z = st["types"]
        mbbp.mbbp_sample_errors(st["n"], case["batch"], 0, st["seed"], case["p"], mbbp.NOISE_DEPOLARIZING,
                                X["e"], Z["e"])
        outs = []
        for t in (X, Z):
            o = t["out"]
            mbbp.mbbp_syndrome(t["B"], t["e"], t["s"])
            mbbp.mbbp_decode(t["B"], t["s"], st["llr"], case["iters"], case["alpha"], mbbp.RULE_NMS, o["e_hat"],
                             o["conv"], o["success"], st["ws"], iters_run=o["iters_run"], selected=o["selected"])
            t["counts"].zero_()
            mbbp.mbbp_judge(t["L"], t["e"], o["e_hat"], t["fail"], t["counts"])
            outs.append([t["e"], t["s"], t["fail"], t["counts"]] + _decode_outputs(o))
        return outs
    B = st["B"]
    if kind == "train":
        scale = 1.0 / (case["batch"] * B.R * B.n)
        args = (B, st["s"], st["llr"], case["T"], st["w"], st["g"], case["ckpt"], st["etrue"], scale, st["post"])
        mbbp.mbbp_wms_forward(*args, st["loss"], st["ws"], all_iters=True)
        st["gw"].zero_()
        st["gg"].zero_()
        mbbp.mbbp_wms_backward(*args, st["gw"], st["gg"], st["ws"], all_iters=True)
        return [st["post"], st["loss"], st["gw"], st["gg"]]
    o = st["out"]
    if kind == "wms_decode":
        mbbp.mbbp_wms_decode(B, st["s"], st["llr"], case["iters"], case["T"], st["w"], st["g"], o["e_hat"], o["conv"],
                             o["success"], st["ws"], iters_run=o["iters_run"], selected=o["selected"])
    elif kind == "realtime":
        mbbp.mbbp_decode_noalloc(B, st["s"], st["llr"], case["iters"], case["alpha"], mbbp.RULE_NMS, o["e_hat"],
                                 o["conv"], o["success"], iters_run=o["iters_run"], selected=o["selected"])
    else:
        mbbp.mbbp_decode_ex(B, st["s"], st["llr"], case["iters"], st["opt"], o["e_hat"], o["conv"], o["success"],
                            st["ws"], iters_run=o["iters_run"], selected=o["selected"])
    return _decode_outputs(o)


# ----------------------------------------------------------------- work

# n, m and row weight of the named codes' check matrices
_SHAPES = {"bb72": (72, 36, 6), "bb144": (144, 72, 6), "bb288": (288, 144, 6), "gb882": (882, 441, 6)}
# edges of an H^(t) over those of H (its subtree repeats part of the rows)
_REPEAT = 1.15
# iterations to the halting rule (flooding, alpha 0.625), averaged over the
# representations of [[144,12,12]], at marginal error rates; the other codes
# are within a factor of about 1.5
_ITERATIONS = ((0.0, 1.0), (0.0134, 1.5), (0.0267, 3.7), (0.04, 9.5), (0.0534, 20.4), (0.06, 27.5))


def _iterations(p, iters, serial=False):
    xs, ys = zip(*_ITERATIONS)
    k = float(np.interp(p, xs, ys))
    return min(iters, k / 3.0 if serial else k)


def _shape(case):
    if case["code"] == "gb":
        return 2 * case["L"], case["L"], 2 * case["weight"]
    return _SHAPES[case["code"]]


def _decode_work(n, m, dc, R, batch, p, iters, serial=False, soft=False):
    """10 operations per edge update (|q|, two minima updates, sign parity,
    select, normalization, sign; posterior sum and extrinsic); bytes: the
    syndromes (and LLRs) in, estimates, flags, iteration counts and the
    selection out."""
    updates = batch * R * (_REPEAT * m * dc) * _iterations(p, iters, serial)
    nbytes = batch * (m + n + R + 2 * R + 1 + 2) + 4 * n * (batch if soft else 1)
    return {"bytes": float(nbytes), "flops": 10.0 * updates}


def work(case):
    kind, batch, p = case["kind"], case["batch"], case["p"]
    if kind == "mixed":
        parts = [_decode_work(*_SHAPES[name], R, batch, p, case["iters"]) for name, R in MIXED for _ in range(2)]
        return {k: sum(x[k] for x in parts) for k in ("bytes", "flops")}
    n, m, dc = _shape(case)
    R = case["R"]
    if kind == "train":
        # forward: the 10 operations and 4 of weight and damping; adjoint:
        # about twice that
        T, E = case["T"], _REPEAT * m * dc
        nbytes = batch * (m + n / 8) + 4.0 * batch * R * (n + 1) + 4 * 4.0 * R * T * E
        return {"bytes": nbytes, "flops": 42.0 * batch * R * T * E}
    if kind == "montecarlo":
        one = _decode_work(n, m, dc, R, batch, 2.0 * p / 3.0, case["iters"])
        # two error types; the packed errors and judge codes go out as well
        return {"bytes": 2 * (one["bytes"] + batch * (4 * ((n + 31) // 32) + 1)), "flops": 2 * one["flops"]}
    w = _decode_work(n, m, dc, R, batch, p, case["iters"], case.get("schedule") == "serial", case.get("soft", False))
    if kind == "wms_decode":
        w["flops"] *= 1.4
        w["bytes"] += 2 * 4.0 * R * case["T"] * _REPEAT * m * dc
    return w


# ----------------------------------------------------------------- exact values

def _splitmix(state, i):
    mask = (1 << 64) - 1
    z = (state + i * 0x9E3779B97F4A7C15) & mask
    z = ((z ^ (z >> 30)) * 0xBF58476D1CE4E5B9) & mask
    z = ((z ^ (z >> 27)) * 0x94D049BB133111EB) & mask
    return z ^ (z >> 31)


def _subtrees(H, R, seed):
    """The rows that the R representations append to H: maximal subtrees of
    the Tanner graph over root orders 0 (the identity), 1, ... (Fisher-Yates
    shuffles), in creation order without repeats of a check set."""
    m = H.shape[0]
    cols = [np.flatnonzero(H[r]).tolist() for r in range(m)]
    rows = [np.flatnonzero(H[:, v]).tolist() for v in range(H.shape[1])]
    out, seen = [], set()
    for j in range(1024):
        perm = list(range(m))
        if j:
            for d, i in enumerate(range(m - 1, 0, -1)):
                x = _splitmix(seed ^ j, d + 1) % (i + 1)
                perm[i], perm[x] = perm[x], perm[i]
        taken = set()
        for root in perm:
            if root in taken:
                continue
            tree, tested, reached, queue = [], set(), set(), [root]
            for u in queue:
                if u in tested:
                    continue
                tested.add(u)
                if sum(v in reached for v in cols[u]) > 1:
                    continue
                tree.append(u)
                taken.add(u)
                for v in cols[u]:
                    reached.add(v)
                    queue.extend(c for c in rows[v] if c not in tested and c not in taken)
            if frozenset(tree) not in seen:
                seen.add(frozenset(tree))
                out.append(tree)
                if len(out) == R:
                    return out
    raise RuntimeError("too few subtrees")


def _exact_train(case, seed):
    """Posteriors, losses and gradients of the weighted min-sum step in 64
    bits, representation by representation."""
    code, g = _code(case), _generator(seed)
    H = code.HZ
    batch, T, R, n = case["batch"], case["T"], case["R"], code.n
    e = _errors(g, batch, n, case["p"])
    s = _syndromes(e, H)
    sets = _subtrees(H, R, BASES_SEED)
    Emax = max(int(H.sum() + H[t].sum()) for t in sets)
    w32, g32 = _weights(g, R, T, Emax)
    mu = _llr(n, case["p"]).double()
    scale = 1.0 / (batch * R * n * T)
    target = e.double()
    post_out = torch.empty((batch, R, n), dtype=torch.float64, device="cuda")
    loss_out = torch.empty((batch, R), dtype=torch.float64, device="cuda")
    gw, gg = (torch.zeros((R, T, Emax), dtype=torch.float64, device="cuda") for _ in range(2))
    for b, tree in enumerate(sets):
        src = list(range(H.shape[0])) + list(tree)
        deg = [int(H[r].sum()) for r in src]
        M, D = len(src), max(deg)
        E = sum(deg)
        var = np.concatenate([np.flatnonzero(H[r]) for r in src])
        slot = np.concatenate([r * D + np.arange(d) for r, d in enumerate(deg)])
        var_t, slot_t = (torch.from_numpy(x).cuda() for x in (var, slot))
        sgn = 1.0 - 2.0 * s[:, src].double()  # [batch, M]
        w = w32[b, :, :E].double().requires_grad_(True)
        d = g32[b, :, :E].double().requires_grad_(True)
        parts = [slice(i, min(batch, i + 1024)) for i in range(0, batch, 1024)]
        for part in parts:
            nb = part.stop - part.start
            m = torch.zeros((nb, E), dtype=torch.float64, device="cuda")
            q = mu[var_t].expand(nb, E)
            loss = 0.0
            for t in range(T):
                dense = torch.full((nb, M * D), LMAX, dtype=torch.float64, device="cuda")
                dense = dense.index_copy(1, slot_t, q).view(nb, M, D)
                mag, sign = dense.abs(), torch.where(dense < 0, -1.0, 1.0).to(torch.float64)
                # smallest and second smallest |q| of each row
                v1, i1 = mag.min(-1, keepdim=True)
                v2 = mag.scatter(-1, i1, math.inf).amin(-1, keepdim=True)
                own = torch.arange(D, device="cuda") == i1
                low = torch.where(own, v2, v1).clamp(max=LMAX)
                par = sign.prod(-1, keepdim=True) * sgn[part].unsqueeze(-1)
                c = (par * sign * low).reshape(nb, M * D).index_select(1, slot_t)
                m = d[t] * m + (1.0 - d[t]) * w[t] * c
                post = mu + torch.zeros((nb, n), dtype=torch.float64, device="cuda").index_add(1, var_t, m)
                q = post.index_select(1, var_t) - m
                x = torch.where(target[part] > 0, post, -post)
                loss = loss + torch.nn.functional.softplus(x, threshold=1e9).sum(-1)
            loss = scale * loss
            loss.sum().backward()
            post_out[part, b] = post.detach()
            loss_out[part, b] = loss.detach()
        gw[b, :, :E], gg[b, :, :E] = w.grad, d.grad
    return [post_out, loss_out, gw, gg]


def exact(case, seed):
    """Training in 64 bits; every other kind returns bits, flags, counts and
    indices only, which have to be equal."""
    if case["kind"] != "train":
        return None
    if work(case)["flops"] > 1.1 * max(work(x)["flops"] for x in listed() if x["kind"] == "train"):
        return None  # over 20 seconds
    return _exact_train(case, seed)
