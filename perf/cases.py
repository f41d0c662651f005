"""The workloads a user of the screening engine runs, as measurable cases.

A case is a dict of plain values.  ``listed()`` names the standing cases,
``draw(rng)`` gives one more of the same ranges, ``prepare(case, seed)`` makes
what a user's program holds before the call (inputs, and the built space or
batch where the program keeps one), ``run(state)`` makes one pass through the
package's public calls and returns everything they produce, ``work(case)`` is
what a pass cannot do without and ``exact(case, seed)`` is the same result from
plain FP64 numpy / torch arithmetic, without this package.

Kinds: ``screen`` (SIS screen of a built space, or of a space built in the
pass), ``loop`` (space build and the residual loop), ``batch`` (re-screen of
many problems with new targets), ``l0`` (exhaustive subset search).
"""
import math

import numpy as np
import torch

from paper_2602_06986_gb300 import dse

SQUARE, CUBE, INV, SQRT, EXP, LOG, ADD, SUB, MUL, DIV, RDIV, ABSDIFF = range(12)
FULL = (1 << 12) - 1
#: + - * / ^2 sqrt exp log
BASIC = FULL & ~((1 << CUBE) | (1 << INV) | (1 << ABSDIFF))
FMAX, FMIN_STD, TAU = 1e15, 1e-8, 1e-10


def _screen(name, n, p, dims, targets, k, precision="auto", mode="per_target", rung=2, ops="full", values="lognormal",
            build=False, host=False, dedup=False, begin=0.0, length=0):
    c = dict(kind="screen", n=n, p=p, dims=dims, targets=targets, k=k, precision=precision, mode=mode, rung=rung,
             ops=ops, values=values, build=build, host=host, dedup=dedup, begin=begin, length=length)
    return dict(c, name=name) if name else c


def _loop(name, n, p, dims, k, iters):
    c = dict(kind="loop", n=n, p=p, dims=dims, k=k, iters=iters, rung=2, ops="full", values="lognormal")
    return dict(c, name=name) if name else c


def _batch(name, bases, n_lo, n_hi, p_lo, p_hi, k):
    c = dict(kind="batch", bases=bases, n_lo=n_lo, n_hi=n_hi, p_lo=p_lo, p_hi=p_hi, k=k, rung=2, ops="full")
    return dict(c, name=name) if name else c


def _l0(name, n, p, dims, ids, dim, top):
    c = dict(kind="l0", n=n, p=p, dims=dims, ids=ids, dim=dim, top=top, rung=2, ops="full", values="lognormal")
    return dict(c, name=name) if name else c


def listed():
    return [
        # a first run on a small table (100 materials, 8 properties): host arrays in, space, top-100, host arrays out
        _screen("tiny_project", 100, 8, 3, 1, 100, "fp32", ops="basic", values="uniform", build=True, host=True),
        # one more target screened against a space that is already built; odd sizes
        _screen("small_screen", 333, 13, 3, 1, 50, "fp32"),
        # the ordinary descriptor search: space, then three SIS + least-squares iterations
        _loop("medium_loop", 1000, 20, 4, 1000, 3),
        # several properties ranked together (multi-task SISSO): one list by the aggregated score
        _screen("medium_aggregated", 1000, 20, 4, 4, 1000, "auto", "aggregated"),
        # a screen that returns no two interchangeable descriptors
        _screen("medium_dedup", 1000, 16, 4, 1, 200, "fp32", dedup=True),
        # many samples, one target, a ragged sample count (beyond the single-target Gram range)
        _screen("long_screen", 9973, 24, 5, 1, 2000, "fp32", values="mixed"),
        # a few targets over a ragged sample count
        _screen("multi_ragged", 1531, 22, 4, 7, 500, "bf16x3"),
        # the largest single problem: 20000 samples, 40 primaries, 16 targets, space build included
        _screen("large_step", 20000, 40, 5, 16, 10000, "auto", values="mixed", build=True),
        # one block of a streamed rung-3 space (sharded or resumed search), 64 targets
        _screen("rung3_block", 500, 12, 0, 64, 1000, "auto", rung=3, values="wide", begin=0.37, length=40_000_001),
        # cross-validation folds and bootstrap resamples of 32 data sets, re-screened with new targets
        _batch("batch_folds", 32, 63, 5000, 10, 30, 200),
        # exhaustive pairs over the union of three SIS subspaces
        _l0("l0_pairs", 1000, 20, 4, 3000, 2, 16),
        # the plain FP64 screen (a user's cross-check of a result)
        _screen("fp64_screen", 500, 10, 3, 1, 200, "fp64"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    most = _cost(listed()[7])
    while True:
        what = rng.choice(["project", "screen", "screen", "aggregated", "dedup", "long", "multi", "multi", "rung3", "loop",
                           "batch", "l0", "fp64"])
        k = _log_int(rng, 20, 4000)
        if what == "project":
            c = _screen("", _log_int(rng, 50, 2000), rng.randint(6, 24), rng.randint(2, 5), 1, min(k, 100), "fp32",
                        ops=rng.choice(["basic", "full"]), values=rng.choice(["uniform", "lognormal"]), build=True,
                        host=rng.random() < 0.5)
        elif what == "screen":
            c = _screen("", _log_int(rng, 50, 2048), rng.randint(8, 28), rng.randint(2, 5), 1, k, "fp32",
                        values=rng.choice(["lognormal", "mixed"]))
        elif what == "aggregated":
            c = _screen("", _log_int(rng, 100, 4000), rng.randint(8, 24), rng.randint(3, 5), rng.randint(2, 8),
                        min(k, 1000), "auto", "aggregated")
        elif what == "dedup":
            c = _screen("", _log_int(rng, 100, 2000), rng.randint(8, 20), rng.randint(3, 5), 1, min(k, 300), "fp32",
                        dedup=True)
        elif what == "long":
            c = _screen("", _log_int(rng, 2049, 20000), rng.randint(8, 30), rng.randint(3, 5), 1, k, "fp32",
                        values="mixed")
        elif what == "multi":
            c = _screen("", _log_int(rng, 200, 20000), rng.randint(10, 40), rng.randint(3, 5), rng.randint(2, 16),
                        _log_int(rng, 100, 10000), "bf16x3", values=rng.choice(["lognormal", "mixed"]),
                        build=rng.random() < 0.5)
        elif what == "rung3":
            c = _screen("", _log_int(rng, 100, 1000), rng.randint(8, 12), 0, rng.choice([17, 32, 48, 64]),
                        min(k, 1000), "auto", rung=3, values="wide", begin=round(rng.uniform(0.05, 0.9), 4),
                        length=_log_int(rng, 100_000, 40_000_000) | 1)
        elif what == "loop":
            c = _loop("", _log_int(rng, 100, 4000), rng.randint(8, 24), rng.randint(3, 5), min(k, 2000), rng.randint(2, 4))
        elif what == "batch":
            lo = _log_int(rng, 63, 300)
            c = _batch("", rng.randint(2, 32), lo, lo * rng.randint(2, 16), 8, rng.randint(12, 30), min(k, 400))
        elif what == "l0":
            dim = rng.randint(1, 3)
            c = _l0("", _log_int(rng, 100, 4000), rng.randint(12, 20), rng.randint(3, 4),
                    _log_int(rng, 100, 700 if dim == 3 else 4000), dim, rng.randint(4, 32))
        else:
            c = _screen("", _log_int(rng, 60, 1000), rng.randint(6, 14), rng.randint(3, 4), 1, min(k, 500), "fp64")
        if _cost(c) <= most and (c["kind"] != "screen" or c["k"] * 4 < _counts(c)[3]):
            return c


# --- inputs -----------------------------------------------------------------

def _ops(case):
    return BASIC if case["ops"] == "basic" else FULL


def _units(p, dims):
    """Unit exponents belong to the data set's columns: the same for every draw of its values."""
    g = np.random.Generator(np.random.PCG64(40_000 + 97 * p + dims))
    return g.integers(-2, 3, size=(p, dims)).astype(np.int32)


def _f32(a):
    return np.asarray(a, np.float32).astype(np.float64)


def _X(g, p, n, values):
    if values == "uniform":
        return g.uniform(0.5, 2.0, (p, n))  # full FP64 values
    if values == "wide":
        return _f32(g.uniform(0.1, 10.0, (p, n)))
    if values == "five":
        return _f32(g.uniform(0.5, 5.0, (p, n)))
    if values == "mixed":
        a, b = (p + 2) // 3, (p + 1) // 3
        return _f32(np.concatenate([g.uniform(0.5, 5.0, (a, n)), g.lognormal(0.0, 0.5, (b, n)),
                                    g.standard_normal((p - a - b, n))]))
    return _f32(g.lognormal(0.0, 0.5, (p, n)))


def _Y(g, X, T):
    """Planted products, sums and quotients of three columns with 1% noise."""
    Z, Y = np.abs(X) + 0.1, np.empty((T, X.shape[1]))
    for t in range(T):
        a, b, c = g.choice(len(Z), 3, replace=False)
        f = (Z[a] * Z[b] / Z[c], (Z[a] + Z[b]) * Z[c], np.sqrt(Z[a]) * Z[b] - Z[c], Z[a] / (Z[b] + Z[c]))[t % 4]
        Y[t] = f + 0.01 * f.std() * g.standard_normal(len(f))
    return Y


def _problem(case, seed):
    g = np.random.Generator(np.random.PCG64([seed, 1]))
    X = _X(g, case["p"], case["n"], case["values"])
    return X, _units(case["p"], case["dims"]), _Y(g, X, case.get("targets", 1)), g


def _problems(case, seed):
    """Per base data set 5 cross-validation folds and 3 bootstrap resamples: (X, units, sample list, target)."""
    fixed = np.random.Generator(np.random.PCG64(case["bases"] * 7 + case["n_hi"]))
    g = np.random.Generator(np.random.PCG64([seed, 2]))
    out = []
    for b in range(case["bases"]):
        n = int(round(math.exp(fixed.uniform(math.log(case["n_lo"]), math.log(case["n_hi"])))))
        n = case["n_lo"] if b == 0 else case["n_hi"] if b == 1 else n
        p = int(fixed.integers(case["p_lo"], case["p_hi"] + 1))
        X = _X(g, p, n, "five")
        y = _Y(g, X, 1)[0]
        folds = np.array_split(g.permutation(n), 5)
        rows = [np.sort(np.concatenate(folds[:f] + folds[f + 1:])) for f in range(5)]
        rows += [np.sort(g.integers(0, n, n)) for _ in range(3)]
        out += [(X, _units(p, 3), r.astype(np.int64), y[r]) for r in rows]
    return out


def _space(case, X, units):
    return dse.Space(X, units, _ops(case), case["rung"])


def prepare(case, seed):
    if case["kind"] == "batch":
        todo = _problems(case, seed)
        spaces = [dse.Space(torch.from_numpy(X).cuda(), u, _ops(case), 2, sample_idx=r) for X, u, r, _ in todo]
        ys = [y for *_, y in todo]
        # the plan is made with a first target (here the samples' first column); the pass brings the real ones
        batch = dse.Batch(spaces, [np.ascontiguousarray(X[0, r]) for X, _, r, _ in todo], case["k"])
        return dict(case=case, batch=batch, Y=torch.from_numpy(np.concatenate(ys)).cuda())
    X, units, Y, g = _problem(case, seed)
    s = dict(case=case, units=units, X=X, Y=Y)
    if not case.get("host"):
        s["X"], s["Y"] = torch.from_numpy(X).cuda(), torch.from_numpy(Y).cuda()
    if case["kind"] == "loop":
        s["sis"] = torch.zeros(case["iters"], case["k"], dtype=torch.int64, device="cuda")
        s["residual"] = torch.zeros(case["n"], dtype=torch.float64, device="cuda")
        return s
    if case["kind"] == "l0":
        s["space"] = _space(case, s["X"], units)
        s["ids"] = torch.from_numpy(_l0_ids(case, s["space"].n_stored, g).astype(np.int64)).cuda()
        return s
    if not case["build"]:
        s["space"] = _space(case, s["X"], units)
        s["range"] = _range(case, s["space"].n_stored, s["space"].n_total)
    if not case["host"]:
        lists = 1 if case["mode"] == "aggregated" else case["targets"]
        s["out"] = [torch.zeros(lists, case["k"], dtype=t, device="cuda")
                    for t in (torch.int64, torch.float64, torch.float64)]
    return s


def _range(case, n_stored, n_total):
    """A block of the last rung's ids at a relative offset, or everything."""
    if not case["length"]:
        return 0, 0
    begin = n_stored + int(case["begin"] * (n_total - n_stored))
    return begin, min(n_total, begin + case["length"])


def _l0_ids(case, n_stored, g):
    """Distinct products and quotients of two stored features, as a list of SIS subspaces holds them."""
    unary, p = sum(1 for o in range(6) if _ops(case) >> o & 1), case["p"]
    pairs = n_stored * (n_stored - 1) // 2 - p * (p - 1) // 2  # pairs of two primaries belong to rung 1
    ids = n_stored + unary * (n_stored - p) + 6 * g.choice(pairs, case["ids"], replace=False)
    return ids + g.integers(MUL - ADD, RDIV - ADD + 1, len(ids))


# --- one pass ---------------------------------------------------------------

PRECISION = {"fp32": dse.PREC_FP32, "fp64": dse.PREC_FP64, "bf16x3": dse.PREC_BF16X3, "auto": dse.PREC_AUTO}


def run(s):
    case = s["case"]
    if case["kind"] == "batch":
        s["batch"].rescreen(s["Y"])
        got = [s["batch"].fetch(i) for i in range(len(s["batch"].spaces))]
        out = [np.zeros((len(got), case["k"]), t) for t in (np.int64, np.float64, np.float64)]
        for i, lst in enumerate(got):
            for o, v in zip(out, lst):
                o[i, :len(v)] = v
        return dict(zip(("ids", "scores", "bounds"), out))
    if case["kind"] == "loop":
        space = _space(case, s["X"], s["units"])
        r = space.residual_loop(s["Y"][0], case["iters"], case["k"], sis_ids=s["sis"], residual=s["residual"])
        size = [space.n_stored, space.n_total]
        space.free()
        return dict(chosen=r["chosen"], rmse=r["rmse"], coefs=r["coefs"], sis=s["sis"], residual=s["residual"], size=size)
    if case["kind"] == "l0":
        pos, rmse, coefs = s["space"].l0_search(s["Y"][0], s["ids"], case["dim"], case["top"])
        return dict(pos=pos, rmse=rmse, coefs=coefs)
    space = _space(case, s["X"], s["units"]) if case["build"] else s["space"]
    begin, end = s.get("range", (0, 0))
    res = space.screen(s["Y"], case["k"], dse.MODE_AGGREGATED if case["mode"] == "aggregated" else dse.MODE_PER_TARGET,
                       PRECISION[case["precision"]], begin, end, dedup_tau=TAU if case["dedup"] else None)
    if case["host"]:
        ids, scores, bounds = res.fetch(0)
        ids = ids.astype(np.int64)
    else:
        ids, scores, bounds = s["out"]
        for t in range(res.n_lists):
            res.fetch(t, out=(ids[t], scores[t], bounds[t]))
    out = dict(ids=ids, scores=scores, bounds=bounds, size=[space.n_stored, space.n_total])
    res.free()
    if case["build"]:
        space.free()
    return out


# --- what a pass cannot do without ------------------------------------------

def _rows(case):
    """(samples, primaries, dims, times) of the case's problems."""
    if case["kind"] != "batch":
        return [(case["n"], case["p"], case["dims"], 1)]
    fixed = np.random.Generator(np.random.PCG64(case["bases"] * 7 + case["n_hi"]))
    out = []
    for b in range(case["bases"]):
        n = int(round(math.exp(fixed.uniform(math.log(case["n_lo"]), math.log(case["n_hi"])))))
        n = case["n_lo"] if b == 0 else case["n_hi"] if b == 1 else n
        out.append((n, int(fixed.integers(case["p_lo"], case["p_hi"] + 1)), 3, 8))
    return out


def _next_rung(u, first, ops):
    """Unit rows of the unit-valid candidates over u, whose rows from `first` on are the newest rung."""
    new = u[first:]
    free = (new == 0).all(1)
    out = [f for o, f in ((SQUARE, 2 * new), (CUBE, 3 * new), (INV, -new), (SQRT, new // 2), (EXP, 0 * new[free]),
                          (LOG, 0 * new[free])) if ops >> o & 1]
    for i in range(first, len(u)):
        same = (u[:i] == u[i]).all(1)
        out += [f for o, f in ((MUL, u[i] + u[:i]), (DIV, u[i] - u[:i]), (RDIV, u[:i] - u[i]), (ADD, u[:i][same]),
                               (SUB, u[:i][same]), (ABSDIFF, u[:i][same])) if ops >> o & 1]
    return np.concatenate(out)


_COUNTED = {}


def _counts(case):
    """(stored features, their samples, slots, unit-valid candidates, their samples) over all problems, by units alone."""
    total = np.zeros(5)
    for n, p, dims, times in _rows(case):
        key = (p, dims, case["rung"], case["ops"])
        if key not in _COUNTED:
            ops = _ops(case)
            u = _units(p, dims).astype(np.int64) << case["rung"]
            first = 0
            for r in range(1, case["rung"]):
                if dims == 0:  # every slot is valid: only the number matters
                    new = len(u) - first
                    pairs = len(u) * (len(u) - 1) // 2 - first * (first - 1) // 2
                    grown = np.zeros((6 * new + 6 * pairs, 0), np.int64)
                else:
                    grown = _next_rung(u, first, ops)
                u, first = np.concatenate([u, grown]), len(u)
            new, o = len(u) - first, first
            pairs = len(u) * (len(u) - 1) // 2 - o * (o - 1) // 2
            _, size = np.unique(u, axis=0, return_counts=True) if dims else (None, np.array([len(u)]))
            _, old = np.unique(u[:o], axis=0, return_counts=True) if dims else (None, np.array([o]))
            same = int((size * (size - 1) // 2).sum() - (old * (old - 1) // 2).sum())
            free = int((u[o:] == 0).all(1).sum())
            bit = [ops >> b & 1 for b in range(12)]
            valid = sum(bit[:4]) * new + sum(bit[4:6]) * free + sum(bit[8:11]) * pairs + (bit[6] + bit[7] + bit[11]) * same
            slots = sum(bit[:6]) * new + sum(bit[6:]) * pairs
            _COUNTED[key] = (len(u), slots, valid)
        stored, slots, valid = _COUNTED[key]
        if case.get("length"):
            valid, slots = valid * min(1.0, case["length"] / slots), min(case["length"], slots)
        else:
            valid += stored
        total += [stored * times, stored * n * times, slots * times, valid * times, valid * n * times]
    return [float(t) for t in total]


def _cost(case):
    """Candidate-sample operations of a pass (FP64 ones counted at their rate)."""
    stored, _, _, valid, vn = _counts(case)
    if case["kind"] == "l0":
        return 64 * (case["ids"] ** 2 / 2 * case["n"] + 12.0 * math.comb(case["ids"], case["dim"]))
    per = 4 if case["kind"] == "batch" else 3 + case.get("targets", 1)
    return vn * per * case.get("iters", 1) * (4 if case.get("dedup") else 1) * (64 if case.get("precision") == "fp64" else 1)


def work(case):
    """Bytes: the primaries and targets in, the lists out.  Flops: per valid candidate and sample one evaluation, two
    moments and one product with each target (l0: the Gram matrix, and one elimination step per subset)."""
    _, _, _, _, vn = _counts(case)
    if case["kind"] == "l0":
        n, m, d = case["n"], case["ids"], case["dim"]
        return dict(bytes=8.0 * n * (case["p"] + 1) + 8.0 * m + case["top"] * 8.0 * (2 * d + 2),
                    flops=1.0 * m * (m + 1) * n + 2.0 * d * d * math.comb(m, d))
    if case["kind"] == "batch":
        rows = _rows(case)
        return dict(bytes=sum(8.0 * n * (p + 8) + 8 * case["k"] * 24.0 for n, p, _, _ in rows), flops=6.0 * vn)
    T = case.get("targets", 1)
    lists = case.get("iters", 1) if case["kind"] == "loop" else 1 if case["mode"] == "aggregated" else T
    width = 8.0 if case["kind"] == "loop" else 24.0
    return dict(bytes=8.0 * case["n"] * (case["p"] + T) + width * lists * case["k"],
                flops=vn * (4.0 + 2.0 * T) * case.get("iters", 1))


# --- the same in 64 bits ----------------------------------------------------

class _Exact:
    """The candidate space in plain FP64 on the device: stored rungs as rows, the last rung by id."""

    def __init__(self, X, units, ops, rung):
        self.V, self.U = torch.zeros(0, X.shape[1], dtype=torch.float64, device="cuda"), np.zeros((0, units.shape[1]), np.int64)
        self.un, self.bi = [o for o in range(6) if ops >> o & 1], [o for o in range(6, 12) if ops >> o & 1]
        rows = torch.from_numpy(X).cuda()
        keep = self._realised(rows).cpu().numpy()
        self._store(rows[torch.from_numpy(keep).cuda()], units[keep].astype(np.int64) << rung)
        self.first = 0
        for _ in range(1, rung):
            n_slots, grown, units_of = self.slots(), [], []
            for lo in range(0, n_slots, 1 << 17):
                v, ok, op, a, b = self.block(lo, min(n_slots, lo + (1 << 17)))
                grown.append(v[ok])
                op, a, b = (t[ok].cpu().numpy() for t in (op, a, b))
                A, B, w = self.U[a], self.U[np.maximum(b, 0)], op[:, None]
                units_of.append(np.select([w == SQUARE, w == CUBE, w == INV, w == SQRT, (w == EXP) | (w == LOG), w == MUL,
                                           w == DIV, w == RDIV], [2 * A, 3 * A, -A, A // 2, 0 * A, A + B, A - B, B - A], A))
            first = len(self.V)
            self._store(torch.cat(grown), np.concatenate(units_of))
            self.first = first

    @staticmethod
    def _realised(v):
        mean = v.mean(1, keepdim=True)
        std = ((v - mean) ** 2).mean(1).sqrt()
        return torch.isfinite(v).all(1) & (std > FMIN_STD * (v * v).mean(1).sqrt())

    def _store(self, rows, units):
        self.V, self.U = torch.cat([self.V, rows]), np.concatenate([self.U, units])
        self.lo, self.hi = self.V.min(1).values, self.V.max(1).values
        self.least, self.most = self.V.abs().min(1).values, self.V.abs().max(1).values
        key = np.unique(self.U, axis=0, return_inverse=True)[1] if self.U.shape[1] else np.zeros(len(self.U), np.int64)
        self.key = torch.from_numpy(key.reshape(-1)).cuda()
        self.free = torch.from_numpy((self.U == 0).all(1)).cuda()

    def slots(self):
        n, o = len(self.V), self.first
        return len(self.un) * (n - o) + len(self.bi) * (n * (n - 1) // 2 - o * (o - 1) // 2)

    def block(self, lo, hi):
        """Values, validity, op and operands of the last rung's flat slots [lo, hi)."""
        o, split = self.first, len(self.un) * (len(self.V) - self.first)
        f = torch.arange(lo, hi, device="cuda")
        is_un = f < split
        q = torch.where(is_un, 0, f - split)
        pair = torch.div(q, len(self.bi), rounding_mode="floor") + o * (o - 1) // 2
        i = ((1 + (1 + 8 * pair.double()).sqrt()) / 2).long()
        i = i - (i * (i - 1) // 2 > pair).long()
        i = i + ((i + 1) * i // 2 <= pair).long()
        a = torch.where(is_un, o + f // len(self.un), i)
        b = torch.where(is_un, -1, pair - i * (i - 1) // 2)
        op = torch.where(is_un, torch.tensor(self.un, device="cuda")[f % len(self.un)], torch.tensor(self.bi, device="cuda")[q % len(self.bi)])
        return self.evaluate(op, a, b) + (op, a, b)

    def evaluate(self, op, a, b):
        c = b.clamp_min(0)
        A, B, ok = self.V[a], self.V[c], torch.ones(len(a), dtype=torch.bool, device="cuda")
        v = torch.zeros_like(A)
        Ma, Mb, ma, mb = self.most[a], self.most[c], self.least[a], self.least[c]
        inf = torch.full_like(Ma, math.inf)

        def slot(code, value, unit_ok, bound):
            m = op == code
            if bool(m.any()):
                v[m] = value(A[m], B[m])
                ok[m] = unit_ok[m] & (bound[m] <= FMAX)

        yes, free, same = torch.ones_like(ok), self.free[a], self.key[a] == self.key[c]
        slot(SQUARE, lambda x, y: x * x, yes, Ma * Ma)
        slot(CUBE, lambda x, y: x * x * x, yes, Ma * Ma * Ma)
        slot(INV, lambda x, y: 1 / x, ma > 0, 1 / ma)
        slot(SQRT, lambda x, y: x.sqrt(), self.lo[a] >= 0, Ma.sqrt())
        slot(EXP, lambda x, y: x.exp(), free & (self.hi[a] <= 80), torch.where(self.hi[a] <= math.log(FMAX), 0 * Ma, inf))
        slot(LOG, lambda x, y: x.log(), free & (self.lo[a] > 0), 0 * Ma)
        slot(ADD, lambda x, y: x + y, same, Ma + Mb)
        slot(SUB, lambda x, y: x - y, same, Ma + Mb)
        slot(MUL, lambda x, y: x * y, yes, Ma * Mb)
        slot(DIV, lambda x, y: x / y, mb > 0, Ma / mb)
        slot(RDIV, lambda x, y: y / x, ma > 0, Mb / ma)
        slot(ABSDIFF, lambda x, y: (x - y).abs(), same, Ma + Mb)
        return v, ok & self._realised(v)

    def columns(self, ids):
        """Value rows of candidate ids (all valid)."""
        out = torch.empty(len(ids), self.V.shape[1], dtype=torch.float64, device="cuda")
        n = len(self.V)
        for r, g in enumerate(ids.tolist()):
            out[r] = self.V[g] if g < n else self.block(g - n, g - n + 1)[0][0]
        return out

    def top(self, Y, k, aggregated=False, begin=0, end=0):
        """Scores and ids of the k best candidates per list."""
        n = len(self.V)
        end = end or n + self.slots()
        Yc = Y - Y.mean(1, keepdim=True)
        Yc = Yc / Yc.norm(dim=1, keepdim=True)
        best = None
        step = max(1, (1 << 28) // self.V.shape[1])
        edges = sorted({begin, end, *range(begin, end, step)} | ({n} if begin < n < end else set()))
        for lo, hi in zip(edges, edges[1:]):
            v, ok = (self.V[lo:hi], torch.ones(hi - lo, dtype=torch.bool, device="cuda")) if hi <= n else \
                self.block(lo - n, hi - n)[:2]
            v, ids = v[ok], torch.arange(lo, hi, device="cuda")[ok]
            v = v - v.mean(1, keepdim=True)
            s = ((v @ Yc.T) / v.norm(dim=1, keepdim=True)).abs().T
            s = (s * s).mean(0, keepdim=True).sqrt() if aggregated else s
            if best is not None:
                s, ids = torch.cat([best[0], s], 1), torch.cat([best[1], ids.expand(len(s), -1)], 1)
            else:
                ids = ids.expand(len(s), -1)
            at = s.topk(min(k, s.shape[1]), 1).indices
            best = s.gather(1, at), ids.gather(1, at)
        return best


def _lists(scores, k):
    out = torch.zeros(len(scores), k, dtype=torch.float64, device="cuda")
    out[:, :scores.shape[1]] = scores
    return out


def _fit(y, cols):
    """Least squares with intercept: coefficients and residual."""
    A = torch.cat([torch.ones_like(y)[None], cols]).T
    q, r = torch.linalg.qr(A)
    beta = torch.linalg.solve_triangular(r, (q.T @ y)[:, None], upper=True)[:, 0]
    return beta, y - A @ beta


def _exact_loop(case, E, y):
    rmse, coefs, chosen, res = [], [], [], y
    for _ in range(case["iters"]):
        _, ids = E.top(res[None], case["k"])
        ids = ids[0][~torch.isin(ids[0], torch.tensor(chosen, device="cuda", dtype=torch.int64))]
        c = E.columns(ids)
        c = c - c.mean(1, keepdim=True)
        raw = c.norm(dim=1)
        basis = torch.ones_like(y)[None] / math.sqrt(len(y))
        if chosen:
            f = E.columns(torch.tensor(chosen))
            basis = torch.cat([basis, torch.linalg.qr((f - f.mean(1, keepdim=True)).T)[0].T])
        for _ in range(2):
            c = c - (c @ basis.T) @ basis
        gain = torch.where(c.norm(dim=1) > 1e-12 * raw, (c @ res) ** 2 / (c * c).sum(1), torch.zeros_like(raw))
        chosen.append(int(ids[gain.argmax()]))
        beta, res = _fit(y, E.columns(torch.tensor(chosen)))
        rmse.append(float((res * res).mean().sqrt()))
        coefs.append([float(b) for b in beta])
    return dict(chosen=None, rmse=rmse, coefs=coefs, sis=None, residual=res, size=None)


def _exact_l0(case, E, y, ids):
    c = E.columns(torch.from_numpy(ids))
    n = len(ids)
    raw = c.norm(dim=1)
    z = c - c.mean(1, keepdim=True)
    yc = y - y.mean()
    G, b = z @ z.T, z @ yc
    raw2 = raw * raw * 1e-24
    best_q, best_s = torch.zeros(0, device="cuda", dtype=torch.float64), torch.zeros(0, case["dim"], device="cuda", dtype=torch.int64)

    def keep(q, s):
        nonlocal best_q, best_s
        q, s = torch.cat([best_q, q]), torch.cat([best_s, s])
        at = q.topk(min(64, len(q))).indices
        best_q, best_s = q[at], s[at]

    one = torch.arange(n, device="cuda")
    d = G.diagonal()
    if case["dim"] == 1:
        keep(torch.where(d > raw2, b * b / d, -1.0), one[:, None])
    for i in range(n if case["dim"] > 1 else 0):  # eliminate i, then rank the rest
        if d[i] <= raw2[i]:
            continue
        g = G[i, i + 1:] / d[i]
        dj, bj, j = d[i + 1:] - g * G[i, i + 1:], b[i + 1:] - g * b[i], one[i + 1:]
        ok = dj > raw2[i + 1:]
        if case["dim"] == 2:
            keep(torch.where(ok, b[i] ** 2 / d[i] + bj * bj / dj, -1.0), torch.stack([j * 0 + i, j], 1))
            continue
        H = G[i + 1:, i + 1:] - g[:, None] * G[i, i + 1:][None]
        r = H / dj[:, None]
        dk, bk = dj[None] - r * H, bj[None] - r * bj[:, None]
        ok = ok[:, None] & (dk > raw2[None, i + 1:]) & (one[:n - i - 1, None] < one[None, :n - i - 1])
        q = torch.where(ok, b[i] ** 2 / d[i] + (bj * bj / dj)[:, None] + bk * bk / dk, -1.0).reshape(-1)
        q, at = q.topk(min(64, len(q))) if len(q) else (q, q.long())
        keep(q, torch.stack([at * 0 + i, i + 1 + at // max(1, n - i - 1), i + 1 + at % max(1, n - i - 1)], 1))
    # interchangeable columns tie, so the RMSEs are determined and the coefficients are not
    rmse = sorted(float(_fit(y, c[t])[1].square().mean().sqrt()) for t in best_s)[:case["top"]]
    return dict(pos=None, rmse=torch.tensor(rmse, dtype=torch.float64), coefs=None)


def exact(case, seed):
    if _cost(case) / (64 if case.get("precision") == "fp64" or case["kind"] == "l0" else 1) > 4e12:
        return None  # minutes in FP64
    if case["kind"] == "batch":
        todo = _problems(case, seed)
        if _counts(case)[4] > 1.5e10 or len(todo) > 64:
            return None
        out = torch.zeros(len(todo), case["k"], dtype=torch.float64, device="cuda")
        for i, (X, u, r, y) in enumerate(todo):
            s = _Exact(np.ascontiguousarray(X[:, r]), u, _ops(case), 2).top(torch.from_numpy(y)[None].cuda(), case["k"])[0]
            out[i, :s.shape[1]] = s[0]
        return dict(ids=None, scores=out, bounds=None)
    X, units, Y, g = _problem(case, seed)
    Y = torch.from_numpy(Y).cuda()
    E = _Exact(X, units, _ops(case), case["rung"])
    if case["kind"] == "loop":
        return _exact_loop(case, E, Y[0])
    if case["kind"] == "l0":
        return _exact_l0(case, E, Y[0], _l0_ids(case, len(E.V), g))
    begin, end = _range(case, len(E.V), len(E.V) + E.slots())
    k = case["k"]
    s, ids = E.top(Y, 20 * k if case["dedup"] else k, case["mode"] == "aggregated", begin, end)
    if case["dedup"]:  # drop every candidate that an interchangeable one of a smaller id precedes
        z = E.columns(ids[0])
        z = z - z.mean(1, keepdim=True)
        z = z / z.norm(dim=1, keepdim=True)
        twin = ((z @ z.T).abs() >= 1 - TAU) & (ids[0][None] < ids[0][:, None])
        s = s[:, ~twin.any(1)][:, :k]
    out = _lists(s, k)
    return dict(ids=None, scores=out[0, :s.shape[1]] if case["host"] else out, bounds=None, size=None)
