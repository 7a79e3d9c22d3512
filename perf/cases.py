"""The work that users of this package have it do, as cases that can be timed and checked.

Every case goes through the Python entry points (`tcorr.Tcorr`, `Batch`, `Server`, `Mp2`,
`task_energy_noalloc`).  Sizes are those of the package's own configurations, tests, profiles and
benchmark: single problems from o=4, v=20 to o=50, v=450, batches of molecules with o in 4..16 and
v in 20..120, served requests with o in 4..40 and v in 20..300, RI-MP2 up to o=50, v=450,
naux=1500.  Inputs follow the package's synthetic recipe (three-index factors of standard deviation
0.1, sorted orbital energies, MP1 doubles, singles of 1e-3), drawn and contracted on the GPU.

A case's `kind`:
  energy    the whole E(T) of a problem whose handle the program keeps
  range     a contiguous share of the task list of a large problem, with per-task energies
  oneshot   create a handle, take E(T), close it: each molecule seen once
  noalloc   one task through the allocation-free entry point
  batch     E(T) of many molecules of uneven size in one handle
  serve     requests submitted to a running server and drained
  mp2       the RI-MP2 energy of a problem whose handle the program keeps
"""
import math

import numpy as np
import torch

from paper_1609_08094_gb300 import tcorr

DEV = "cuda:0"


def listed():
    return [
        # the smallest configuration in FP64: launches and latency
        {"name": "fp64_energy_o4_v20", "kind": "energy", "prec": "fp64", "o": 4, "v": 20, "naux": 72},
        # one FP64 task for a caller whose device memory is its own pool; ragged v
        {"name": "noalloc_task_o8_v61", "kind": "noalloc", "prec": "fp64", "o": 8, "v": 61, "naux": 207},
        # a screening loop: each small molecule is set up, evaluated once and dropped
        {"name": "oneshot_bf16x3_o10_v100", "kind": "oneshot", "prec": "bf16x3", "o": 10, "v": 100, "naux": 330},
        # an ordinary problem of odd sizes, whole energy, in TF32 split precision
        {"name": "energy_tf32x3_o13_v131", "kind": "energy", "prec": "tf32x3", "o": 13, "v": 131, "naux": 432},
        # a worker's share of the large configuration's task list, in each mixed precision
        {"name": "range_bf16x3_o50_v450", "kind": "range", "prec": "bf16x3", "o": 50, "v": 450, "naux": 1500,
         "first": 9001, "count": 28},
        {"name": "range_tf32x3_o50_v450", "kind": "range", "prec": "tf32x3", "o": 50, "v": 450, "naux": 1500,
         "first": 9001, "count": 28},
        # the same in FP64 emulation, at the largest served size
        {"name": "range_fp64oz_o40_v300", "kind": "range", "prec": "fp64_oz", "o": 40, "v": 300, "naux": 1020,
         "first": 4003, "count": 52},
        # the large configuration on the FP64 pipe: one task
        {"name": "range_fp64_o50_v450", "kind": "range", "prec": "fp64", "o": 50, "v": 450, "naux": 1500,
         "first": 9001, "count": 1},
        # molecules of uneven size evaluated together
        {"name": "batch_bf16x3_24", "kind": "batch", "prec": "bf16x3", "n": 24, "o_min": 4, "o_max": 16,
         "v_min": 20, "v_max": 120, "sizes": 4},
        # a burst of requests of uneven size served from submission to the last result
        {"name": "serve_bf16x3_8", "kind": "serve", "prec": "bf16x3",
         "shapes": "4x20 9x64 14x41 27x77 6x180 11x120 17x97 5x300"},
        # RI-MP2 of the large system in the paper's mixed-precision variant, and a smaller one in FP64
        {"name": "mp2_bf16x3_o50_v450", "kind": "mp2", "prec": "bf16x3", "o": 50, "v": 450, "naux": 1500},
        {"name": "mp2_fp64_o16_v256", "kind": "mp2", "prec": "fp64", "o": 16, "v": 256, "naux": 816},
    ]


def _log_int(rng, lo, hi):
    return min(hi, int(math.exp(rng.uniform(math.log(lo), math.log(hi + 1)))))


def _tasks(o):
    return o * (o + 1) * (o + 2) // 6


# Work bounds of drawn cases, in contraction flops of one pass: what a pass of a listed case of the
# same kind and precision costs at most.
_MOST = {"fp64": 4e11, "fp64_oz": 5e12, "tf32x3": 1.2e13, "bf16x3": 1.4e13}


def draw(rng):
    kind = rng.choice(["energy", "energy", "range", "range", "oneshot", "noalloc", "batch", "serve", "mp2"])
    if kind == "noalloc":
        o, v = rng.randint(2, 40), _log_int(rng, 9, 64)
        return {"kind": kind, "prec": "fp64", "o": o, "v": v, "naux": 3 * (o + v)}
    if kind == "mp2":
        prec = rng.choice(["fp64", "tf32x3", "bf16x3"])
        while True:
            o, v = _log_int(rng, 4, 50), _log_int(rng, 20, 450)
            naux = min(1500, 3 * (o + v))
            if prec != "fp64" or tcorr.mp2_flops(o, v, naux) <= 1e11:
                return {"kind": kind, "prec": prec, "o": o, "v": v, "naux": naux}
    if kind == "batch":
        return {"kind": kind, "prec": rng.choice(["tf32x3", "bf16x3", "fp64_oz"]), "n": rng.randint(4, 24), "o_min": 4,
                "o_max": 16, "v_min": 20, "v_max": 120, "sizes": rng.randrange(1 << 20)}
    if kind == "serve":
        shapes, left = [], 7e12
        for _ in range(rng.randint(3, 10)):
            o, v = rng.randint(4, 40), _log_int(rng, 20, 300)
            f = 12.0 * v ** 3 * (v + o) * (_tasks(o) - o)
            if f <= left:
                shapes.append("%dx%d" % (o, v))
                left -= f
        shapes = shapes or ["4x%d" % _log_int(rng, 20, 120)]
        return {"kind": kind, "prec": rng.choice(["tf32x3", "bf16x3"]), "shapes": " ".join(shapes)}
    prec = rng.choice(["fp64", "fp64_oz", "tf32x3", "bf16x3", "bf16x3"])
    if kind == "range":
        while True:
            o, v = _log_int(rng, 12, 50), _log_int(rng, 100, 450)
            per = 12.0 * v ** 3 * (v + o)
            if prec == "fp64_oz" and v ** 3 * o > 1.2e9:
                continue
            count = min(200, _tasks(o) // 2, int(_MOST[prec] / per))
            if count >= 1:
                count = rng.randint(max(1, count // 3), count)
                return {"kind": kind, "prec": prec, "o": o, "v": v, "naux": min(1500, 3 * (o + v)),
                        "first": rng.randint(0, _tasks(o) - count), "count": count}
    most = 2e12 if kind == "energy" else 3e11
    while True:
        o, v = rng.randint(3, 24), _log_int(rng, 16, 300)
        if 12.0 * v ** 3 * (v + o) * (_tasks(o) - o) <= min(most, _MOST[prec]):
            return {"kind": kind, "prec": prec, "o": o, "v": v, "naux": 3 * (o + v)}


# ---- inputs ---------------------------------------------------------------------------------------

def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed) & 0x7FFFFFFFFFFFFFFF)


def _energies(o, v, g):
    eo = torch.sort(-2.0 + 1.7 * torch.rand(o, dtype=torch.float64, device=DEV, generator=g)).values
    ev = torch.sort(0.1 + 4.9 * torch.rand(v, dtype=torch.float64, device=DEV, generator=g)).values
    return eo, ev


def _problem(o, v, naux, seed):
    """(eps_occ, eps_vir, t1, t2, vvvo, ooov, ovov) of one synthetic system.  The factor products are
    formed in FP32 and scaled by sigma^2 in FP64, so that every value has a full FP64 significand."""
    g = _gen(seed)
    n = o + v
    eo, ev = _energies(o, v, g)
    t1 = 1e-3 * torch.randn(o, v, dtype=torch.float64, device=DEV, generator=g)
    B = torch.randn(naux, n, n, dtype=torch.float32, device=DEV, generator=g)
    B = torch.triu(B)
    B = B + torch.triu(B, 1).transpose(1, 2)
    ov = B[:, :o, o:].reshape(naux, o * v)
    oo = B[:, :o, :o].reshape(naux, o * o)
    vo = B[:, o:, :o].reshape(naux, v * o)
    vv = B[:, o:, o:].reshape(naux, v * v)
    del B
    ovov = (ov.T @ ov).double().mul_(0.005)
    ovov = (ovov + ovov.T).reshape(o, v, o, v)
    ooov = (oo.T @ ov).double().mul_(0.01).reshape(o, o, o, v)
    vvvo = torch.empty(v * v, v * o, dtype=torch.float64, device=DEV)
    rows = max(1, (1 << 28) // (v * o))
    for r in range(0, v * v, rows):
        vvvo[r:r + rows].copy_(vv[:, r:r + rows].T @ vo).mul_(0.01)
    d = eo[:, None, None, None] + eo[None, None, :, None] - ev[None, :, None, None] - ev[None, None, None, :]
    t2 = (ovov / d).permute(0, 2, 1, 3).contiguous()
    return eo, ev, t1, t2, vvvo.reshape(v, v, v, o), ooov, ovov


def _mp2_problem(o, v, naux, seed):
    g = _gen(seed)
    eo, ev = _energies(o, v, g)
    return eo, ev, 0.1 * torch.randn(naux, v, o, dtype=torch.float64, device=DEV, generator=g)


def _shapes(case):
    if case["kind"] == "serve":
        return [tuple(int(x) for x in s.split("x")) for s in case["shapes"].split()]
    r = np.random.RandomState(case["sizes"])
    return [(int(r.randint(case["o_min"], case["o_max"] + 1)), int(r.randint(case["v_min"], case["v_max"] + 1)))
            for _ in range(case["n"])]


def _problems(case, seed):
    return [(o, v, *_problem(o, v, 3 * (o + v), seed * 1009 + m)) for m, (o, v) in enumerate(_shapes(case))]


def _task_of(case, seed):
    """The noalloc case's task: three different occupied orbitals where there are as many."""
    o = case["o"]
    i = seed % max(1, o - 2)
    return (i, min(i + 1, o - 1), o - 1)


def prepare(case, seed):
    kind = case["kind"]
    if kind in ("batch", "serve"):
        probs = _problems(case, seed)
        if kind == "batch":
            return {"kind": kind, "handle": tcorr.Batch(probs, prec=case["prec"])}
        return {"kind": kind, "handle": tcorr.Server(prec=case["prec"]), "problems": probs}
    o, v, naux = case["o"], case["v"], case["naux"]
    if kind == "mp2":
        return {"kind": kind, "handle": tcorr.Mp2(o, v, naux, *_mp2_problem(o, v, naux, seed), prec=case["prec"])}
    arrays = _problem(o, v, naux, seed)
    if kind == "oneshot":
        return {"kind": kind, "o": o, "v": v, "arrays": arrays, "prec": case["prec"]}
    if kind == "noalloc":
        return {"kind": kind, "o": o, "v": v, "arrays": arrays, "ijk": _task_of(case, seed),
                "out": torch.zeros(2, dtype=torch.float64, device=DEV)}
    st = {"kind": kind, "handle": tcorr.Tcorr(o, v, *arrays, prec=case["prec"])}
    if kind == "range":
        st["first"], st["count"] = case["first"], case["count"]
    big = arrays[4].numel() > 1 << 28
    del arrays  # the handle keeps its own layouts: a program with a large problem frees the inputs
    if big:
        torch.cuda.empty_cache()
    return st


def run(state):
    kind = state["kind"]
    if kind == "energy":
        return np.array(state["handle"].energy())
    if kind == "range":
        e, tasks = state["handle"].energy_range(state["first"], state["count"], per_task=True)
        return {"e": np.array(e), "tasks": tasks}
    if kind == "oneshot":
        with tcorr.Tcorr(state["o"], state["v"], *state["arrays"], prec=state["prec"]) as t:
            return np.array(t.energy())
    if kind == "noalloc":
        tcorr.task_energy_noalloc(state["o"], state["v"], *state["arrays"], state["ijk"], state["out"])
        return state["out"]
    if kind == "batch":
        return state["handle"].energy()
    if kind == "serve":
        server = state["handle"]
        ids = [server.submit(p) for p in state["problems"]]
        server.drain()
        got = [server.poll(j) for j in ids]
        bad = [g for g in got if g[0] != "done"]
        if bad:
            raise RuntimeError("served job not done: %r" % (bad[0],))
        return np.array([g[1] for g in got])
    return np.array(state["handle"].energy())


def work(case):
    """Bytes: every input array in FP64 read once (of a task share or a single task: what its tasks
    read of it) and the energies written; for a kept handle its own operands are of that size or
    more.  Flops: 12 v^3 (v + o) per task (2 v^2 naux per RI-MP2 pair)."""
    kind = case["kind"]

    def one(o, v):
        b = 8.0 * (o + v + o * v + 2 * (o * v) ** 2 + v ** 3 * o + o ** 3 * v)
        return b, 12.0 * v ** 3 * (v + o) * (_tasks(o) - o)

    if kind in ("batch", "serve"):
        got = [one(o, v) for o, v in _shapes(case)]
        return {"bytes": sum(b for b, _ in got) + 24.0 * len(got), "flops": sum(f for _, f in got)}
    o, v = case["o"], case["v"]
    if kind == "mp2":
        return {"bytes": 8.0 * (o + v + o * v * case["naux"]) + 24, "flops": tcorr.mp2_flops(o, v, case["naux"])}
    if kind == "noalloc":
        ijk = _task_of(case, 1)
        some = len(set(ijk)) > 1
        return {"bytes": 8.0 * (3 * v ** 3 + 3 * o * v * v + 6 * v * v + 9 * o * v + 2),
                "flops": 12.0 * v ** 3 * (v + o) if some else 1.0}
    if kind == "range":
        tasks = _task_list(o)[case["first"]:case["first"] + case["count"]]
        occ = len({x for t in tasks for x in t})
        busy = sum(1 for t in tasks if t[0] != t[2])
        return {"bytes": 8.0 * occ * (v ** 3 + o * v * v * 2) + 16.0 * len(tasks),
                "flops": max(1.0, 12.0 * v ** 3 * (v + o) * busy)}
    b, f = one(o, v)
    return {"bytes": b + 24, "flops": f}


# ---- the same results in 64 bits, in plain torch ---------------------------------------------------

def _task_list(o):
    return [(i, j, k) for i in range(o) for j in range(i, o) for k in range(j, o)]


class _Reference:
    """E[4] and E[5] of single tasks, from the equations over the ordered occupied triples."""

    def __init__(self, o, v, eo, ev, t1, t2, vvvo, ooov, ovov):
        self.o, self.v, self.eo, self.ev, self.t1, self.t2 = o, v, eo, ev, t1, t2
        self.vvvo, self.ooov, self.ovov = vvvo, ooov, ovov
        self.slices = {}

    def _slice(self, k):
        if k not in self.slices:
            if len(self.slices) * self.v ** 3 > 4e9:
                self.slices.clear()
            self.slices[k] = self.vvvo[:, :, :, k].contiguous().reshape(self.v, self.v * self.v)  # [d][b c]
        return self.slices[k]

    def _w(self, i, j, k):
        # w^{abc}_{ijk} = sum_d t^{ad}_{ij} (bd|ck) - sum_l t^{ab}_{il} (ck|lj), (bd|ck) = (db|ck)
        v, o = self.v, self.o
        w = (self.t2[i, j] @ self._slice(k)).reshape(v, v, v)
        ll = self.ooov[:, j, k, :]                                    # (lj|kc)
        w -= (self.t2[i].reshape(o, v * v).T @ ll).reshape(v, v, v)
        return w

    def task(self, i, j, k):
        if i == k:
            return 0.0, 0.0
        W = self._w(i, j, k)
        W += self._w(i, k, j).permute(0, 2, 1)
        W += self._w(j, i, k).permute(1, 0, 2)
        W += self._w(j, k, i).permute(2, 0, 1)
        W += self._w(k, i, j).permute(1, 2, 0)
        W += self._w(k, j, i).permute(2, 1, 0)
        t1, g, ev = self.t1, self.ovov, self.ev
        Y = t1[i][:, None, None] * g[j, :, k, :][None, :, :]
        Y = Y + t1[j][None, :, None] * g[i, :, k, :][:, None, :]
        Y = Y + t1[k][None, None, :] * g[i, :, j, :][:, :, None]
        D = self.eo[i] + self.eo[j] + self.eo[k] - ev[:, None, None] - ev[None, :, None] - ev[None, None, :]
        R = W / D
        # the orderings of (i, j, k) are permutations of (a, b, c) of the same W, Y and D
        A = torch.zeros_like(W)
        for p in ((0, 1, 2), (0, 2, 1), (1, 0, 2), (1, 2, 0), (2, 0, 1), (2, 1, 0)):
            Rp = R.permute(p)
            # the sum of x~ R over this ordering, with the tilde's three terms moved onto R
            A += (4.0 * Rp - 6.0 * Rp.permute(0, 2, 1) + 2.0 * Rp.permute(1, 2, 0)).permute(
                tuple(int(x) for x in np.argsort(p))) / 3.0
        m = (6 if i < j < k else 3) / 6.0
        return m * float((A * W).sum()), m * float((A * Y).sum())


def _energies_of(ref, tasks):
    e = np.array([ref.task(*t) for t in tasks]).reshape(-1, 2)
    return e, np.array([math.fsum(e[:, 0]), math.fsum(e[:, 1]), math.fsum(e.reshape(-1))])


def exact(case, seed):
    kind = case["kind"]
    allow = torch.backends.cuda.matmul.allow_tf32
    torch.backends.cuda.matmul.allow_tf32 = False
    try:
        if kind in ("batch", "serve"):
            return np.array([_energies_of(_Reference(*p), _task_list(p[0]))[1] for p in _problems(case, seed)])
        o, v, naux = case["o"], case["v"], case["naux"]
        if kind == "mp2":
            return _exact_mp2(o, v, *_mp2_problem(o, v, naux, seed))
        ref = _Reference(o, v, *_problem(o, v, naux, seed))
        if kind == "noalloc":
            return torch.tensor(ref.task(*_task_of(case, seed)), dtype=torch.float64)
        if kind == "range":
            e, total = _energies_of(ref, _task_list(o)[case["first"]:case["first"] + case["count"]])
            return {"e": total, "tasks": e}
        return _energies_of(ref, _task_list(o))[1]
    finally:
        torch.backends.cuda.matmul.allow_tf32 = allow


def _exact_mp2(o, v, eo, ev, C):
    Ct = C.permute(2, 1, 0).contiguous()                              # [i][a][gamma]
    ej, ek = [], []
    for i in range(o):
        for j in range(i, o):
            G = Ct[i] @ Ct[j].T                                       # g_aibj
            X = G / (ev[:, None] + ev[None, :] - eo[i] - eo[j])
            w = 1.0 if i == j else 2.0
            ej.append(-2.0 * w * (X * G).sum())
            ek.append(w * (X * G.T).sum())
    ej, ek = math.fsum(torch.stack(ej).tolist()), math.fsum(torch.stack(ek).tolist())
    return np.array([ej, ek, ej + ek])
