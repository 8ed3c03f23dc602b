"""Kernel variants chosen by the shape of the call, each against the FP32
oracle bit for bit (normalized min-sum) at the sizes where a variant can go
wrong: the last partly filled block of rows, rows that do not fill the kernel
width, calls with and without posteriors.
"""
import numpy as np
import pytest

import oracle
from paper_2605_14170_gb300.inputs import channel_llr, gb_code, named_code

pytestmark = pytest.mark.gpu

SEED = 20260601


def _decode(B, s, llr, iters, alpha, **kw):
    import torch
    from paper_2605_14170_gb300 import mbbp
    out = mbbp.decode(B, torch.from_numpy(np.ascontiguousarray(s)).cuda(),
                      torch.from_numpy(np.ascontiguousarray(llr, np.float32)).cuda(), iters, alpha, **kw)
    torch.cuda.synchronize()
    res = {k: v.cpu().numpy() for k, v in out.items() if k not in ("cand", "workspace")}
    res["iters"] = res["iters"].view(np.uint16)
    res["cand"] = mbbp.unpack_words(out["cand"], B.n)
    return res


def _assert_exact(got, ref):
    for key, rkey in (("conv", "conv"), ("iters", "iters"), ("cand", "cand"), ("selected", "selected"),
                      ("success", "success"), ("e_hat", "ehat")):
        assert np.array_equal(got[key], ref[rkey]), key


def _irregular(m, n, wmax, seed):
    """Rows of weight 2..wmax, every column of weight 1..3."""
    rng = np.random.default_rng(seed)
    H = np.zeros((m, n), np.uint8)
    H[np.arange(n) % m, np.arange(n)] = 1
    for r in range(m):
        want = int(rng.integers(2, wmax + 1))
        free = [v for v in rng.permutation(n) if H[r, v] == 0 and H[:, v].sum() < 3]
        for v in free[:max(0, want - int(H[r].sum()))]:
            H[r, v] = 1
    return H


CODES = {
    # width 6, every row full, more variables than the small-code shapes take
    "gb166": lambda: gb_code(83, [0, 7, 31], [2, 19, 55]).HZ,
    # width 8 (rows of weight 8), width 12 (rows of weight 10)
    "gb90w4": lambda: gb_code(45, [0, 3, 11, 30], [1, 8, 20, 37]).HZ,
    "gb78w5": lambda: gb_code(39, [0, 3, 11, 21, 30], [1, 8, 20, 27, 36]).HZ,
    # width 6 with rows of several weights
    "irregular": lambda: _irregular(70, 190, 6, 5),
}


@pytest.mark.parametrize("post", [False, True])
@pytest.mark.parametrize("code", sorted(CODES))
def test_generic_flooding_variants(code, post):
    """The generic flooding kernel's variants: rows that fill the width or
    not, outputs with posteriors or without."""
    from paper_2605_14170_gb300 import mbbp
    H = CODES[code]()
    n = H.shape[1]
    e, _ = oracle.sample(SEED, 0, 65, n, 0.04, "bsc")
    s = oracle.syndrome(H, e)
    llr = channel_llr(n, 0.04).astype(np.float32)
    B = mbbp.mbbp_build_bases(H, 5, SEED)
    got = _decode(B, s, llr, 40, 0.7, want_posterior=post)
    _assert_exact(got, oracle.mbbp_decode(H, B.sets, s, llr, 40, 0.7, precision="f32"))


@pytest.mark.parametrize("code", ["gb78w5", "irregular12"])
def test_serial_width_12(code):
    """The serial schedule's kernel of width 12 (tables of its own, rows in their
    own order): rows of 10 and rows of weight 2 to 12, outputs and posteriors
    bit for bit as the FP32 oracle's."""
    import torch
    from paper_2605_14170_gb300 import mbbp
    H = _irregular(50, 150, 12, 7) if code == "irregular12" else CODES[code]()
    n, R = H.shape[1], 4
    e, _ = oracle.sample(SEED + 12, 0, 41, n, 0.03, "bsc")
    s = oracle.syndrome(H, e)
    llr = np.random.default_rng(13).uniform(1.0, 3.0, n).astype(np.float32)
    B = mbbp.mbbp_build_bases(H, R, SEED)
    out = _decode(B, s, llr, 30, 0.7, schedule=mbbp.SCHEDULE_SERIAL, want_posterior=True)
    _assert_exact(out, oracle.mbbp_decode(H, B.sets, s, llr, 30, 0.7, precision="f32",
                                          schedule=oracle.SCHEDULE_SERIAL))
    ref = [[oracle.bp(np.vstack([H, H[rows]]), np.concatenate([x, x[rows]]), llr, 30, 0.7, precision="f32",
                      schedule=1)["post"] for rows in B.sets] for x in s]
    assert np.array_equal(out["posterior"], np.array(ref))


@pytest.mark.parametrize("iters", [0, 1, 40])
@pytest.mark.parametrize("code", sorted(CODES))
def test_generic_posteriors(code, iters):
    """Posteriors of the generic flooding kernels, which hold them by position
    until an item ends, by variable as the FP32 oracle has them: bit for bit,
    alone and together with the message trace."""
    import torch
    from paper_2605_14170_gb300 import mbbp
    H = CODES[code]()
    n, R = H.shape[1], 3
    e, _ = oracle.sample(SEED + 11, 0, 17, n, 0.04, "bsc")
    s = oracle.syndrome(H, e)
    llr = np.random.default_rng(12).uniform(1.0, 3.0, n).astype(np.float32)
    B = mbbp.mbbp_build_bases(H, R, SEED)
    ref = np.stack([[oracle.bp(np.vstack([H, H[rows]]), np.concatenate([x, x[rows]]), llr, iters, 0.7,
                               precision="f32")["post"] for rows in B.sets] for x in s])
    for trace in (False, True):
        out = mbbp.decode(B, torch.from_numpy(s).cuda(), torch.from_numpy(llr).cuda(), iters, 0.7,
                          want_posterior=True, want_c2v=trace)
        torch.cuda.synchronize()
        assert np.array_equal(out["posterior"].cpu().numpy(), ref), trace


@pytest.mark.parametrize("schedule", ["flooding", "serial"])
@pytest.mark.parametrize("code", ["bb72", "irregular"])
def test_empty_row(code, schedule):
    """A matrix with a row without entries, in H and in a repeated set."""
    from paper_2605_14170_gb300 import mbbp
    H = (named_code("bb72").HZ if code == "bb72" else CODES[code]()).copy()
    H[5] = 0
    sets, n = [[0], [1, 5, 9], [2, 3]], H.shape[1]
    e, _ = oracle.sample(SEED + 9, 0, 33, n, 0.04, "bsc")
    s = oracle.syndrome(H, e)
    llr = channel_llr(n, 0.04).astype(np.float32)
    B = mbbp.mbbp_build_bases_from_sets(H, sets)
    sched = (mbbp.SCHEDULE_SERIAL, oracle.SCHEDULE_SERIAL) if schedule == "serial" else (mbbp.SCHEDULE_FLOODING,
                                                                                       oracle.SCHEDULE_FLOODING)
    got = _decode(B, s, llr, 20, 0.7, schedule=sched[0])
    _assert_exact(got, oracle.mbbp_decode(H, sets, s, llr, 20, 0.7, precision="f32", schedule=sched[1]))


@pytest.mark.parametrize("ckpt,all_iters", [(1, True), (3, False), (7, True)])
@pytest.mark.parametrize("code", ["bb72", "gb90w4", "gb78w5", "irregular"])
def test_wms_training_one_shot_per_lane(code, ckpt, all_iters):
    """129 shots at R = 3: the training kernels with one shot per lane (shared
    LLRs; a last block of one shot) against the warp-per-shot kernels, which
    the same LLRs given per shot take.  Same posteriors bit for bit; losses
    and gradients to the rounding of their sums: two orders of N terms differ
    by at most 2 N 2^-24 sum|terms| (the losses' terms are of one sign and
    added in partial sums of at most 42: 1e-5; the gradients', by norm:
    1e-4)."""
    import torch
    from paper_2605_14170_gb300 import mbbp
    H = named_code("bb72").HZ if code == "bb72" else CODES[code]()
    n, T, batch, R = H.shape[1], 7, 129, 3
    e, _ = oracle.sample(SEED + 1, 0, batch, n, 0.05, "bsc")
    s = torch.from_numpy(oracle.syndrome(H, e)).cuda()
    B = mbbp.mbbp_build_bases(H, R, SEED)
    rng = np.random.default_rng(3)
    E = int(B.edges.max())
    w, g = (torch.from_numpy(rng.uniform(lo, hi, (R, T, E)).astype(np.float32)).cuda()
            for lo, hi in ((0.4, 1.0), (0.0, 0.4)))
    mu = torch.from_numpy(rng.uniform(1.0, 3.5, n).astype(np.float32)).cuda()
    et = torch.from_numpy(mbbp.pack_bits(e)).cuda()
    res = []
    for llr in (mu, mu.repeat(batch, 1).contiguous()):
        post = torch.full((batch, R, n), 7.0, device="cuda")
        loss = torch.full((batch, R), 7.0, device="cuda")
        gw, gg = torch.zeros_like(w), torch.zeros_like(g)
        ws = torch.empty(mbbp.mbbp_wms_workspace_size(B, batch, T, ckpt), dtype=torch.uint8, device="cuda")
        mbbp.mbbp_wms_forward(B, s, llr, T, w, g, ckpt, et, 1e-3, post, loss, ws, all_iters=all_iters)
        mbbp.mbbp_wms_backward(B, s, llr, T, w, g, ckpt, et, 1e-3, post, gw, gg, ws, all_iters=all_iters)
        torch.cuda.synchronize()
        res.append([x.double().cpu().numpy() for x in (post, loss, gw, gg)])
    (p1, l1, w1, g1), (p2, l2, w2, g2) = res
    assert np.array_equal(p1, p2)
    assert np.allclose(l1, l2, rtol=1e-5, atol=0)
    for a, b in ((w1, w2), (g1, g2)):
        assert np.linalg.norm(b) > 0
        assert np.linalg.norm(a - b) <= 1e-4 * np.linalg.norm(b)


@pytest.mark.parametrize("ckpt,all_iters", [(1, False), (3, True), (6, True)])
@pytest.mark.parametrize("code", ["bb72", "gb90w4", "irregular"])
def test_wms_training_odd_variable_classes(code, ckpt, all_iters):
    """87 shots at R = 3 (the kernels with one shot per lane), representations
    with an odd number of variables of some degree: the step that such a
    class fills by half adds to no variable twice.  Gradients against the
    FP64 oracle's adjoint by norm: 1e-3 bounds FP32 rounding and the odd
    near-tie of two minima, a variable counted twice moves the norm by one
    part in sqrt(n) at least (5e-2 here)."""
    import torch
    from paper_2605_14170_gb300 import mbbp
    H = named_code("bb72").HZ if code == "bb72" else CODES[code]()
    n, T, batch, R, scale = H.shape[1], 6, 87, 3, 1e-3
    e, _ = oracle.sample(SEED + 5, 0, batch, n, 0.05, "bsc")
    s = oracle.syndrome(H, e)
    B = mbbp.mbbp_build_bases(H, R, SEED)
    degrees = [H.sum(0, dtype=int) + H[rows].sum(0, dtype=int) for rows in B.sets]
    assert any((np.bincount(d) % 2).any() for d in degrees)
    rng = np.random.default_rng(4)
    E = int(B.edges.max())
    w, g = (rng.uniform(lo, hi, (R, T, E)).astype(np.float32) for lo, hi in ((0.4, 1.0), (0.0, 0.4)))
    mu = rng.uniform(1.5, 3.5, n).astype(np.float32)
    ref = [np.zeros((R, T, E)) for _ in range(2)]
    for shot in range(batch):
        for b, rows in enumerate(B.sets):
            Eb = int(B.edges[b])
            grads = oracle.wms_backward(np.concatenate([H, H[rows]]), np.concatenate([s[shot], s[shot][rows]]), mu,
                                        w[b][:, :Eb], g[b][:, :Eb], e[shot], scale, all_iters=all_iters)[1:]
            for r, x in zip(ref, grads):
                r[b][:, :Eb] += x
    wt, gt, st, mt, et = (torch.from_numpy(x).cuda() for x in (w, g, s, mu, mbbp.pack_bits(e)))
    post = torch.empty((batch, R, n), device="cuda")
    gw, gg = torch.zeros_like(wt), torch.zeros_like(gt)
    ws = torch.empty(mbbp.mbbp_wms_workspace_size(B, batch, T, ckpt), dtype=torch.uint8, device="cuda")
    mbbp.mbbp_wms_forward(B, st, mt, T, wt, gt, ckpt, et, scale, post, None, ws, all_iters=all_iters)
    mbbp.mbbp_wms_backward(B, st, mt, T, wt, gt, ckpt, et, scale, post, gw, gg, ws, all_iters=all_iters)
    torch.cuda.synchronize()
    for got, r in zip((gw, gg), ref):
        assert np.linalg.norm(r) > 0
        assert np.linalg.norm(got.double().cpu().numpy() - r) <= 1e-3 * np.linalg.norm(r)


@pytest.mark.parametrize("batch", [20, 300])
def test_wms_checkpoint_interval_beyond_T(batch):
    """A checkpoint interval longer than T needs no more workspace than T
    itself and gives the same gradients (to the order of their sums, as
    above), with the kernels of one shot per lane (300 shots) and of one warp
    per shot (20)."""
    import torch
    from paper_2605_14170_gb300 import mbbp
    H, R, T, n = named_code("bb144").HZ, 8, 6, 144
    e, _ = oracle.sample(SEED + 10, 0, batch, n, 0.05, "bsc")
    s, et = torch.from_numpy(oracle.syndrome(H, e)).cuda(), torch.from_numpy(mbbp.pack_bits(e)).cuda()
    B = mbbp.mbbp_build_bases(H, R, SEED)
    w, g = mbbp.wms_params(B, T, alpha=0.7)
    g += 0.1
    mu = torch.from_numpy(np.random.default_rng(5).uniform(1.0, 3.5, n).astype(np.float32)).cuda()
    assert mbbp.mbbp_wms_workspace_size(B, batch, T, 1000) == mbbp.mbbp_wms_workspace_size(B, batch, T, T)
    res = []
    for ckpt in (2, T, 1000):
        post = torch.empty((batch, R, n), device="cuda")
        gw, gg = torch.zeros_like(w), torch.zeros_like(g)
        ws = torch.empty(mbbp.mbbp_wms_workspace_size(B, batch, T, ckpt), dtype=torch.uint8, device="cuda")
        mbbp.mbbp_wms_forward(B, s, mu, T, w, g, ckpt, et, 1e-3, post, None, ws, all_iters=True)
        mbbp.mbbp_wms_backward(B, s, mu, T, w, g, ckpt, et, 1e-3, post, gw, gg, ws, all_iters=True)
        torch.cuda.synchronize()
        res.append([x.double() for x in (gw, gg)])
    for other in res[1:]:
        for a, b in zip(other, res[0]):
            assert float(b.norm()) > 0 and float((a - b).norm()) <= 1e-4 * float(b.norm())


@pytest.mark.parametrize("shots", [1, 3, 200, 1601])
def test_small_code_run_lengths(shots):
    """The small-code kernel's runs of 8, 2 and 1 shots ([[72]], R = 64: the
    last 16 shots per resident warp come in short runs): one shot, an odd
    batch in runs of 1 and 2, a batch with all three."""
    from paper_2605_14170_gb300 import mbbp
    H = named_code("bb72").HZ
    e, _ = oracle.sample(SEED + 2, 0, shots, 72, 0.05, "bsc")
    s = oracle.syndrome(H, e)
    llr = channel_llr(72, 0.05).astype(np.float32)
    B = mbbp.mbbp_build_bases(H, 64, SEED)
    got = _decode(B, s, llr, 25, 0.625)
    _assert_exact(got, oracle.mbbp_decode(H, B.sets, s, llr, 25, 0.625, precision="f32"))


@pytest.mark.parametrize("code", ["bb72", "bb144"])
def test_small_code_item_per_warp(code):
    """The small-code kernel without work pulls, up to and beyond the most
    items that the resident warps hold at one each (152 SMs x 20 to 24 warps,
    R = 64: 47 to 57 shots); the workspace holds ones, as a call finds it."""
    import torch
    from paper_2605_14170_gb300 import mbbp
    H = named_code(code).HZ
    n = H.shape[1]
    e, _ = oracle.sample(SEED + 8, 0, 64, n, 0.05, "bsc")
    s = oracle.syndrome(H, e)
    llr = channel_llr(n, 0.05).astype(np.float32)
    B = mbbp.mbbp_build_bases(H, 64, SEED)
    ref = oracle.mbbp_decode(H, B.sets, s, llr, 25, 0.625, precision="f32")
    for shots in (1, 40, *range(45, 60), 64):
        ws = torch.full((mbbp.mbbp_decode_workspace_size(B, shots),), 255, dtype=torch.uint8, device="cuda")
        got = {"e_hat": torch.zeros((shots, n), dtype=torch.uint8), "conv": torch.zeros((shots, 64), dtype=torch.uint8),
               "success": torch.zeros(shots, dtype=torch.uint8), "selected": torch.zeros(shots, dtype=torch.int16),
               "iters": torch.zeros((shots, 64), dtype=torch.int16)}
        got = {k: v.cuda() for k, v in got.items()}
        mbbp.mbbp_decode(B, torch.from_numpy(s[:shots]).cuda(), torch.from_numpy(llr).cuda(), 25, 0.625,
                         mbbp.RULE_NMS, got["e_hat"], got["conv"], got["success"], ws, iters_run=got["iters"],
                         selected=got["selected"])
        torch.cuda.synchronize()
        for key, rkey in (("e_hat", "ehat"), ("conv", "conv"), ("success", "success"), ("selected", "selected"),
                          ("iters", "iters")):
            assert np.array_equal(got[key].cpu().numpy(), ref[rkey][:shots]), (key, shots)


@pytest.mark.parametrize("rule", ["nms", "sp"])
@pytest.mark.parametrize("code,R,shots", [("bb72", 64, 2000), ("irregular", 64, 2003), ("gb90w4", 20, 1001),
                                          ("gb166", 8, 1300)])
def test_serial_one_shot_per_lane(code, R, shots, rule):
    """Serial batches long enough for the one-shot-per-lane kernel: slots
    refilled several times, odd layers and variable classes, rows that do not
    fill the width, both widths, zero syndromes among the shots.  Min-sum
    against the FP32 oracle bit for bit; both rules against the warp-per-slot
    kernel (which the same LLRs given per shot take) bit for bit."""
    from paper_2605_14170_gb300 import mbbp
    H = named_code("bb72").HZ if code == "bb72" else CODES[code]()
    n = H.shape[1]
    e, _ = oracle.sample(SEED + 3, 0, shots, n, 0.04, "bsc")
    s = oracle.syndrome(H, e)
    s[::7] = 0
    rng = np.random.default_rng(9)
    llr = rng.uniform(1.0, 4.0, n).astype(np.float32)
    llr[::11] = -0.5
    B = mbbp.mbbp_build_bases(H, R, SEED)
    kw = dict(rule=mbbp.RULE_SP if rule == "sp" else mbbp.RULE_NMS, schedule=mbbp.SCHEDULE_SERIAL)
    got = _decode(B, s, llr, 12, 0.8, **kw)
    ref = _decode(B, s, np.tile(llr, (shots, 1)), 12, 0.8, **kw)
    for key in ("conv", "iters", "cand", "selected", "success", "e_hat"):
        assert np.array_equal(got[key], ref[key]), key
    if rule == "nms":
        _assert_exact(got, oracle.mbbp_decode(H, B.sets, s, llr, 12, 0.8, precision="f32",
                                              schedule=oracle.SCHEDULE_SERIAL))


SERIAL_LIMIT = {
    # code, rows of H repeated in every representation: bytes of shared memory
    # that the one-shot-per-lane layout takes besides 256 of fixed size, of
    # 232448 in all
    "230528": (lambda: gb_code(160, [0, 7, 31], [2, 19, 55]).HZ, lambda H: [list(range(53))] * 64),
    "232320": (lambda: gb_code(144, [76, 90, 106, 132], [56, 104, 112, 138]).HZ,
               lambda H: oracle.collect_subtrees(H, 20, 20260514)),
    "232448": (lambda: gb_code(160, [0, 7, 31], [2, 19, 55]).HZ, lambda H: [list(range(54))] * 64),
}


@pytest.mark.parametrize("size", sorted(SERIAL_LIMIT))
def test_serial_one_shot_per_lane_shared_memory_limit(size):
    """Serial batches of codes on both sides of the shared memory that the
    one-shot-per-lane kernel may take: decoded, bit for bit as by the
    warp-per-slot kernel (which the same LLRs given per shot take) and, for
    the first shots, by the FP32 oracle."""
    from paper_2605_14170_gb300 import mbbp
    code, rows = SERIAL_LIMIT[size]
    H = code()
    n, sets = H.shape[1], rows(H)
    shots = 84_000 // len(sets)
    e, _ = oracle.sample(SEED + 6, 0, shots, n, 0.08, "bsc")
    s = oracle.syndrome(H, e)
    llr = channel_llr(n, 0.08).astype(np.float32)
    B = mbbp.mbbp_build_bases_from_sets(H, sets)
    got = _decode(B, s, llr, 8, 0.8, schedule=mbbp.SCHEDULE_SERIAL)
    ref = _decode(B, s, np.tile(llr, (shots, 1)), 8, 0.8, schedule=mbbp.SCHEDULE_SERIAL)
    for key in ("conv", "iters", "cand", "selected", "success", "e_hat"):
        assert np.array_equal(got[key], ref[key]), key
    few = oracle.mbbp_decode(H, sets, s[:16], llr, 8, 0.8, precision="f32", schedule=oracle.SCHEDULE_SERIAL)
    _assert_exact({k: v[:16] for k, v in got.items()}, few)


SERIAL_BLOCKS = {  # code, R: blocks of the one-shot-per-lane kernel that an SM holds
    "bb72": (lambda: named_code("bb72").HZ, 64),                                # 4
    "gb36w4": (lambda: gb_code(18, [0, 3, 11, 16], [1, 8, 12, 15]).HZ, 8),      # 4, width 8
    "gb100": (lambda: gb_code(50, [0, 7, 31], [2, 19, 44]).HZ, 20),             # 3
    "bb144": (lambda: named_code("bb144").HZ, 64),                              # 2
    "irregular8": (lambda: _irregular(60, 120, 8, 6), 8),                       # 1, width 8
}


@pytest.mark.parametrize("rule,iters", [("nms", 0), ("nms", 9), ("sp", 9)])
@pytest.mark.parametrize("code", sorted(SERIAL_BLOCKS))
def test_serial_one_shot_per_lane_blocks(code, rule, iters):
    """The one-shot-per-lane kernel at each number of blocks per SM, both
    widths, irregular rows, and no iterations at all: 130,000 (shot,
    representation) pairs of random syndromes, which the kernel takes (the
    word behind the candidates says so).  Bit for bit as the warp-per-slot
    kernel and, min-sum, for the first shots as the FP32 oracle."""
    import torch
    from paper_2605_14170_gb300 import mbbp
    make, R = SERIAL_BLOCKS[code]
    H = make()
    n, shots = H.shape[1], 130_000 // R
    e, _ = oracle.sample(SEED + 7, 0, shots, n, 0.4, "bsc")
    s = oracle.syndrome(H, e)
    s[:5] = 0  # halt at once
    llr = np.random.default_rng(8).uniform(0.5, 2.0, n).astype(np.float32)
    B = mbbp.mbbp_build_bases(H, R, SEED)
    kw = dict(rule=mbbp.RULE_SP if rule == "sp" else mbbp.RULE_NMS, schedule=mbbp.SCHEDULE_SERIAL)
    st = torch.from_numpy(s).cuda()
    lanes, slots = (mbbp.decode(B, st, torch.from_numpy(x).cuda(), iters, 0.8, **kw)
                    for x in (llr, np.tile(llr, (shots, 1))))
    torch.cuda.synchronize()
    word = (shots * R * ((n + 31) // 32) * 4 + 255) // 256 * 256
    assert int(lanes["workspace"][word:word + 4].view(torch.int32)) == 1
    for key in ("conv", "iters", "cand", "selected", "success", "e_hat"):
        assert torch.equal(lanes[key], slots[key]), key
    if rule == "nms":
        got = {k: v[:32].cpu().numpy() for k, v in lanes.items() if k != "workspace"}
        got["iters"], got["cand"] = got["iters"].view(np.uint16), mbbp.unpack_words(got["cand"], n)
        _assert_exact(got, oracle.mbbp_decode(H, B.sets, s[:32], llr, iters, 0.8, precision="f32",
                                              schedule=oracle.SCHEDULE_SERIAL))


@pytest.mark.parametrize("p,rounds,lanes", [(0.004, 40, 0), (0.02, 20, 0), (0.08, 20, 1), (0.08, 12, 0)])
def test_serial_route(p, rounds, lanes):
    """The rule of the one-shot-per-lane kernel: at least 16 rounds of 32 items
    per SM and rounds * density^2 * min(1, density / 0.12) >= 0.2 + 0.008 * 20
    iterations (syndrome densities 0.02, 0.11 and 0.32: 0.003, 0.21, 2.1 and,
    too short, 1.2), decided on the device; the result is the oracle's either
    way."""
    import torch
    from paper_2605_14170_gb300 import mbbp
    H, R, n = named_code("bb72").HZ, 64, 72
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    shots = 32 * sms * rounds // R
    e, _ = oracle.sample(SEED + 8, 0, shots, n, p, "bsc")
    s = oracle.syndrome(H, e)
    llr = channel_llr(n, p).astype(np.float32)
    B = mbbp.mbbp_build_bases(H, R, SEED)
    out = mbbp.decode(B, torch.from_numpy(s).cuda(), torch.from_numpy(llr).cuda(), 20, 0.8,
                      schedule=mbbp.SCHEDULE_SERIAL)
    torch.cuda.synchronize()
    word = (shots * R * 3 * 4 + 255) // 256 * 256
    if rounds >= 16:
        assert int(out["workspace"][word:word + 4].view(torch.int32)) == lanes
    ref = oracle.mbbp_decode(H, B.sets, s[:100], llr, 20, 0.8, precision="f32", schedule=oracle.SCHEDULE_SERIAL)
    for key, rkey in (("e_hat", "ehat"), ("conv", "conv"), ("success", "success"), ("selected", "selected")):
        assert np.array_equal(out[key][:100].cpu().numpy(), ref[rkey]), key


@pytest.mark.parametrize("R", [1, 4, 5, 8, 9, 16, 17, 32, 33, 64])
def test_selection_widths(R):
    """Frequency-weighted selection with 4, 8, 16 or 32 lanes per shot (R up to
    32) and beyond, an odd batch; at 0.09 some shots have no candidate and
    some several."""
    from paper_2605_14170_gb300 import mbbp
    H = named_code("bb72").HZ
    e, _ = oracle.sample(SEED + 4, 0, 77, 72, 0.09, "bsc")
    s = oracle.syndrome(H, e)
    llr = channel_llr(72, 0.09).astype(np.float32)
    B = mbbp.mbbp_build_bases(H, R, SEED)
    got = _decode(B, s, llr, 15, 0.625)
    ref = oracle.mbbp_decode(H, B.sets, s, llr, 15, 0.625, precision="f32")
    assert 0 < ref["success"].sum()
    _assert_exact(got, ref)


@pytest.mark.parametrize("L", [6, 30, 48, 80, 81, 159, 160, 162])
def test_syndrome_and_judge_mask_kernels(L):
    """Syndromes and judge codes where the mask kernels' sizes end (160
    variables and 96 rows; 320 and 160) and past them, against the
    definitions."""
    import torch
    from paper_2605_14170_gb300 import mbbp
    code = gb_code(L, [0, 1, 2], [0, 1, 2])  # k = 4 where 3 divides L
    H, n = code.HZ, 2 * L
    batch = 131
    rng = np.random.default_rng(L)
    e = (rng.random((batch, n)) < 0.1).astype(np.uint8)
    ehat = e.copy()
    ehat[::3] ^= (rng.random((len(ehat[::3]), n)) < 0.02).astype(np.uint8)  # mostly wrong syndromes
    ops = mbbp.mbbp_logicals_build(H, code.HX)
    lops = ops.ops()
    flips = mbbp.mbbp_logicals_build(code.HX, H).ops()  # no syndrome, not stabilizers
    assert ops.k == (4 if L % 3 == 0 else 0)
    for i in range(1, batch, 3):  # a check of the other type, or also a logical operator
        ehat[i] ^= code.HX[i % L]
        if ops.k and i % 2:
            ehat[i] ^= flips[i % ops.k]
    sets = [[0]]
    B = mbbp.mbbp_build_bases_from_sets(H, sets)
    ep = torch.from_numpy(mbbp.pack_bits(e)).cuda()
    s = torch.empty((batch, L), dtype=torch.uint8, device="cuda")
    mbbp.mbbp_syndrome(B, ep, s)
    assert np.array_equal(s.cpu().numpy(), (e.astype(int) @ H.T.astype(int) % 2).astype(np.uint8))
    fail = torch.empty(batch, dtype=torch.uint8, device="cuda")
    counts = torch.zeros(3, dtype=torch.int64, device="cuda")
    mbbp.mbbp_judge(ops, ep, torch.from_numpy(ehat).cuda(), fail, counts)
    r = (e ^ ehat).astype(int)
    bad = (r @ H.T.astype(int) % 2).any(1)
    odd = (r @ lops.T.astype(int) % 2).any(1) if ops.k else np.zeros(batch, bool)
    want = np.where(bad, 1, np.where(odd, 2, 0))
    assert bad.any() and not bad.all() and (not ops.k or (want == 2).any())
    assert np.array_equal(fail.cpu().numpy(), want)
    assert np.array_equal(counts.cpu().numpy(), np.bincount(want, minlength=3))
