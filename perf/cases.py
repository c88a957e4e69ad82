"""The calls a program makes to this framework, with sizes: what its speed is measured on.

Each case is one whole call (or the short run of calls a program makes together) through the
public Python entry points; ``prepare`` makes the inputs and the handle that such a program
keeps, ``run`` makes the call, ``exact`` computes the same with plain torch in 64-bit integers.

Kinds of case:

* ``step``: ``Fractal.step`` on a compact state, ``steps`` generations per call (optionally with
  the temporal-blocking option set on the handle).
* ``host``: ``Fractal.run_host``, from pinned host buffers to pinned host buffers.
* ``box``: a compact state scattered into its bounding box, stepped there with
  ``Fractal.bb_step`` and gathered again: the comparison with the bounding-box approach.
* ``maps``: lambda, nu and the compact coordinate of arrays of cells.
* ``batch``: many uneven instances advanced together with ``Batch.run``.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2110_12952_gb300 import Batch, Fractal
from paper_2110_12952_gb300 import workloads as W

#: life-like rules (birth, survive): the 2D and 3D defaults, and others that users of life-like rules run
RULES = {
    "B3/S23": W.LIFE_B3S23,
    "B5/S45": W.MENGER_B5S45,
    "B36/S23": W.rule_masks([3, 6], [2, 3]),
    "B2/S123": W.rule_masks([2], [1, 2, 3]),
    "B4/S345": W.rule_masks([4], [3, 4, 5]),
}

#: levels that calls use, per fractal: from small instances to the largest configured one (the Cantor set, whose
#: cells have no neighbours, is left out: nothing lives there)
LEVELS = {
    "triangle": (6, 20), "carpet": (3, 10), "vicsek": (4, 12), "menger": (3, 7),
    "full_square": (4, 13), "triangle_mirrored": (6, 17),
    "h_fractal": (3, 9), "x_fractal": (4, 11), "chandelier": (4, 13),
    "candy": (3, 7), "empty_bottles": (3, 9),
}
MAIN = ("triangle", "carpet", "vicsek", "menger")
OTHERS = tuple(sorted(set(LEVELS) - set(MAIN)))

MAX_CELLS = 3 ** 20           # the largest configured state
MAX_UPDATES = 3_300_000_000   # cells x generations of a drawn call (the largest listed ones do as many or more)
MAX_BOX = 729 ** 3            # box cells of a drawn bounding-box call
MAX_POINTS = 1 << 25


def _step(name, family, r, steps, p, rule="B3/S23", tb=0):
    return {"name": name, "kind": "step", "family": family, "r": r, "steps": steps, "p": p, "rule": rule, "tb": tb}


def listed():
    return [
        # the smallest configured instance, 100 generations per call: launches and latency
        _step("triangle_r8_x100", "triangle", 8, 100, 0.5),
        # the paper's largest level that still has a bounding box, run for many generations: the state stays in L2
        _step("triangle_r16_x50", "triangle", 16, 50, 0.3),
        # the largest configured state, one generation per call (a program that looks at every generation)
        _step("triangle_r20", "triangle", 20, 1, 0.3),
        # the carpet, one generation per call on a state far larger than L2
        _step("carpet_r10", "carpet", 10, 1, 0.5),
        # the carpet run for many generations per call, with the handle's default settings
        _step("carpet_r9_x20", "carpet", 9, 20, 0.5),
        # the 3D sponge, one generation per call on a state far larger than L2
        _step("menger_r7", "menger", 7, 1, 0.5, "B5/S45"),
        # the configured 3D sponge, run for many generations per call
        _step("menger_r6_x50", "menger", 6, 50, 0.5, "B5/S45"),
        # a fractal of the paper's table that has no kernel of its own
        _step("h_fractal_r9_x4", "h_fractal", 9, 4, 0.5),
        # compact state -> bounding box -> two box generations -> compact state, in three dimensions
        {"name": "box_menger_r6", "kind": "box", "family": "menger", "r": 6, "steps": 2, "p": 0.5, "rule": "B5/S45"},
        # the maps on arrays of cells at the largest level: renderers, samplers, analyses
        {"name": "maps_triangle_r20", "kind": "maps", "family": "triangle", "r": 20, "points": MAX_POINTS - 3},
        # the batched mix: uneven instances of the three 2D fractals advanced together
        {"name": "batch_256", "kind": "batch", "instances": 256, "mix": 7, "steps": 50},
        # one generation from host memory to host memory
        {"name": "host_triangle_r18", "kind": "host", "family": "triangle", "r": 18, "steps": 1, "p": 0.3,
         "rule": "B3/S23"},
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _level(rng, family, most):
    """A level of the family's range with at most `most` cells; levels are a logarithmic scale of sizes."""
    k = W.FAMILIES[family].k
    lo, hi = LEVELS[family]
    while hi > lo and k ** hi > most:
        hi -= 1
    return rng.randint(lo, hi)


def _rule(rng, family, r):
    """A rule under which something lives there for a while."""
    if W.FAMILIES[family].dim == 3:
        return rng.choice(("B5/S45", "B4/S345")) if r >= 5 else "B4/S345"
    return "B2/S123" if family == "x_fractal" else rng.choice(("B3/S23", "B3/S23", "B36/S23", "B2/S123"))


def draw(rng):
    kind = rng.choice(("step",) * 7 + ("box", "box", "maps", "maps", "batch", "host"))
    if kind == "batch":
        return {"kind": "batch", "instances": _log_int(rng, 3, 256), "mix": rng.randrange(1000), "steps": _log_int(rng, 2, 50)}
    family = rng.choice(MAIN * 2 + OTHERS)
    fam = W.FAMILIES[family]
    p = round(rng.uniform(0.3, 0.6), 2)
    if kind == "maps":
        return {"kind": "maps", "family": family, "r": _level(rng, family, MAX_CELLS),
                "points": _log_int(rng, 1000, MAX_POINTS - 1)}
    if kind == "box":
        lo, hi = LEVELS[family]
        while hi > lo and (fam.s ** hi) ** fam.dim > MAX_BOX:
            hi -= 1
        r = rng.randint(lo, hi)
        return {"kind": "box", "family": family, "r": r, "steps": rng.randint(1, 2), "p": p,
                "rule": _rule(rng, family, r)}
    r = _level(rng, family, 3 ** 18 if kind == "host" else MAX_CELLS)
    rule = _rule(rng, family, r)
    if kind == "host":
        return {"kind": "host", "family": family, "r": r, "steps": rng.choice((1, 1, 8)), "p": p, "rule": rule}
    steps = _log_int(rng, 1, max(1, min(100, MAX_UPDATES // fam.k ** r)))
    tb = rng.choice((0, 0, 9, rng.randint(2, 8))) if family in ("carpet", "vicsek") and r >= 3 and steps > 1 else 0
    return {"kind": "step", "family": family, "r": r, "steps": steps, "p": p, "rule": rule, "tb": tb}


# ------------------------------------------------------------------ inputs

def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _bernoulli(cells, p, gen):
    return torch.empty(cells, dtype=torch.uint8, device="cuda").bernoulli_(p, generator=gen)


def _points(case, seed):
    """Cells (omega) and coordinates: those of other cells, moved by at most one along each axis, so that some
    are off the fractal or outside the box, as the neighbours of cells are."""
    fam, n = W.FAMILIES[case["family"]], case["points"]
    gen = _generator(seed)
    omega = torch.randint(0, fam.k ** case["r"], (n,), dtype=torch.int64, device="cuda", generator=gen)
    other = torch.randint(0, fam.k ** case["r"], (n,), dtype=torch.int64, device="cuda", generator=gen)
    move = torch.randint(-1, 2, (n, fam.dim), dtype=torch.int32, device="cuda", generator=gen)
    coords = _Plain(fam, case["r"]).lam(other).to(torch.int32).add_(move)
    return omega, coords


def _mix(case):
    """The instances of a batch: (family, level, p)."""
    return [(i.family, i.r, i.p) for i in W.batched_mix(case["instances"], master_seed=case["mix"])]


def _batch_states(case, seed):
    mix = _mix(case)
    cells = [fam.k ** r for fam, r, _ in mix]
    first = np.concatenate([[0], np.cumsum([(c + 255) // 256 * 256 for c in cells])])
    state = torch.zeros(int(first[-1]), dtype=torch.uint8, device="cuda")
    gen = _generator(seed)
    for (fam, r, p), c, o in zip(mix, cells, first):
        state[int(o):int(o) + c].bernoulli_(p, generator=gen)
    return mix, cells, first, state


def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        mix, cells, first, state = _batch_states(case, seed)
        out = torch.zeros_like(state)
        handles, batch = {}, Batch()
        for (fam, r, _), c, o in zip(mix, cells, first):
            if (fam.name, r) not in handles:
                handles[fam.name, r] = Fractal.from_family(fam, r)
            batch.add(handles[fam.name, r], state[int(o):int(o) + c], out[int(o):int(o) + c], case["steps"])
        return {"kind": kind, "batch": batch, "out": out}
    fam = W.FAMILIES[case["family"]]
    fr = Fractal.from_family(fam, case["r"])
    s = {"kind": kind, "fr": fr}
    if kind == "maps":
        s["omega"], s["coords"] = _points(case, seed)
        return s
    s["rule"], s["steps"] = RULES[case["rule"]], case["steps"]
    s["state"] = _bernoulli(fr.cells, case["p"], _generator(seed))
    if kind == "host":
        s["state"] = s["state"].cpu().pin_memory()
        s["out"] = torch.empty_like(s["state"]).pin_memory()
    elif kind == "box":
        s["box"] = torch.empty(fr.box_cells, dtype=torch.uint8, device="cuda")
        s["box_out"] = torch.empty_like(s["box"])
        s["out"] = torch.empty_like(s["state"])
    else:
        if case["tb"]:
            fr.set_temporal_blocking(case["tb"])
        s["out"] = torch.empty_like(s["state"])
    return s


def run(s):
    kind = s["kind"]
    if kind == "step":
        return s["fr"].step(s["state"], out=s["out"], steps=s["steps"], rule=s["rule"])
    if kind == "host":
        return s["fr"].run_host(s["state"], s["out"], steps=s["steps"], rule=s["rule"])
    if kind == "box":
        fr = s["fr"]
        fr.scatter(s["state"], out=s["box"])
        fr.bb_step(s["box"], out=s["box_out"], steps=s["steps"], rule=s["rule"])
        return {"box": s["box_out"], "compact": fr.gather(s["box_out"], out=s["out"])}
    if kind == "maps":
        fr = s["fr"]
        return {"coords": fr.lam(s["omega"]), "omega": fr.nu(s["coords"]), "compact": fr.nu2d(s["coords"])}
    s["batch"].run()
    return s["out"]


def work(case):
    """Bytes: the state read once and the last generation written once (for a box call the box read and written
    too, for the maps their arrays).  Operations: per cell and generation the neighbours counted and the rule."""
    kind = case["kind"]
    if kind == "batch":
        cells = sum(fam.k ** r for fam, r, _ in _mix(case))
        return {"bytes": 2 * cells, "flops": 10 * cells * case["steps"]}
    fam, r = W.FAMILIES[case["family"]], case["r"]
    cells, nb = fam.k ** r, 3 ** fam.dim + 1
    if kind == "maps":
        n, d = case["points"], fam.dim
        return {"bytes": n * (8 + 4 * d) + n * (4 * d + 8) + n * (4 * d + 8 * d), "flops": n * r * (2 * d + 2)}
    if kind == "box":
        box = (fam.s ** r) ** fam.dim
        # compact in, box out (scatter); box in and out (step); box members in, compact out (gather)
        return {"bytes": 3 * box + 3 * cells, "flops": nb * cells * case["steps"]}
    return {"bytes": 2 * cells, "flops": nb * cells * case["steps"]}


# --------------------------------------------------------- plain computation

class _Plain:
    """lambda, nu and the compact coordinate with plain torch in 64 bits, several levels per table look-up."""

    def __init__(self, fam, r):
        self.k, self.s, self.dim, self.r = fam.k, fam.s, fam.dim, r
        self.off = np.asarray(fam.offsets, dtype=np.int64).reshape(fam.k, fam.dim)
        self.side = fam.s ** r

    def _levels(self, most):
        """(first level, levels) groups whose tables have at most `most` entries."""
        base = max(self.k, self.s ** self.dim)
        m = 1
        while base ** (m + 1) <= most:
            m += 1
        return [(b, min(m, self.r - b)) for b in range(0, self.r, m)]

    def _lam_table(self, m):
        w = np.arange(self.k ** m)
        c = np.zeros((len(w), self.dim), dtype=np.int64)
        for mu in range(m):
            c += self.off[w % self.k] * self.s ** mu
            w = w // self.k
        return c

    def lam(self, omega):
        out = torch.zeros(omega.numel(), self.dim, dtype=torch.int64, device=omega.device)
        for b, m in self._levels(1 << 16):
            t = torch.from_numpy(self._lam_table(m)).to(omega.device)
            out += t[omega // self.k ** b % self.k ** m] * self.s ** b
        return out

    def _index(self, coords, b, m):
        i = torch.zeros(coords.shape[0], dtype=torch.int64, device=coords.device)
        for a in range(self.dim):
            i += coords[:, a] // self.s ** b % self.s ** m * (self.s ** m) ** a
        return i

    def _table(self, m, values):
        """Table over m levels' digits of the coordinates: values(replica digits of the members), -1 elsewhere."""
        w = np.arange(self.k ** m)
        digits = [w // self.k ** mu % self.k for mu in range(m)]
        c = self._lam_table(m)
        i = sum(c[:, a] * (self.s ** m) ** a for a in range(self.dim))
        t = np.full((self.s ** m) ** self.dim, -1, dtype=np.int64)
        t[i] = values(digits)
        return t

    def _inside(self, coords):
        return ((coords >= 0) & (coords < self.side)).all(dim=1)

    def nu(self, coords):
        c = coords.to(torch.int64)
        ok = self._inside(c)
        c = c.clamp(0, self.side - 1)
        out = torch.zeros(c.shape[0], dtype=torch.int64, device=c.device)
        for b, m in self._levels(1 << 16):
            t = self._table(m, lambda d: sum(x * self.k ** mu for mu, x in enumerate(d)))
            h = torch.from_numpy(t).to(c.device)[self._index(c, b, m)]
            ok &= h >= 0
            out += h * self.k ** b
        return torch.where(ok, out, -1)

    def compact(self, coords):
        c = coords.to(torch.int64)
        ok = self._inside(c)
        c = c.clamp(0, self.side - 1)
        out = torch.zeros(c.shape[0], self.dim, dtype=torch.int64, device=c.device)
        for b, m in self._levels(1 << 16):
            i = self._index(c, b, m)
            for a in range(self.dim):
                t = self._table(m, lambda d: sum((x * self.k ** ((b + mu) // self.dim) for mu, x in enumerate(d)
                                                  if (b + mu) % self.dim == a), np.zeros_like(d[0])))
                h = torch.from_numpy(t).to(c.device)[i]
                ok &= h >= 0
                out[:, a] += h
        return torch.where(ok[:, None], out, -1)

    def moves(self):
        return [m for m in np.ndindex(*(3,) * self.dim) if any(x != 1 for x in m)]

    def neighbours(self, lo, hi, device):
        """For each Moore direction the neighbours of cells lo..hi-1; absent ones point one past the state."""
        c = self.lam(torch.arange(lo, hi, dtype=torch.int64, device=device))
        for m in self.moves():
            n = self.nu(c + torch.tensor([x - 1 for x in m], dtype=torch.int64, device=device))
            yield torch.where(n >= 0, n, self.k ** self.r)

    def step(self, state, steps, rule):
        cells, chunk = self.k ** self.r, 1 << 25
        table = torch.zeros(64, dtype=torch.uint8)
        for t in range(32):
            table[t] = rule[0] >> t & 1
            table[32 + t] = rule[1] >> t & 1
        table = table.to(state.device)
        chunks = [(lo, min(lo + chunk, cells)) for lo in range(0, cells, chunk)]
        kept = None
        if steps > 1 and cells * len(self.moves()) * 8 <= 60 << 30:
            kept = [list(self.neighbours(lo, hi, state.device)) for lo, hi in chunks]
        now = torch.cat([(state != 0).to(torch.uint8), torch.zeros(1, dtype=torch.uint8, device=state.device)])
        for _ in range(steps):
            new = torch.zeros_like(now)
            for i, (lo, hi) in enumerate(chunks):
                total = torch.zeros(hi - lo, dtype=torch.uint8, device=state.device)
                for n in kept[i] if kept is not None else self.neighbours(lo, hi, state.device):
                    total += now[n]
                new[lo:hi] = table[(total + 32 * now[lo:hi]).to(torch.int64)]
            now = new
        return now[:-1]


def _too_long(cells, r, steps, dim):
    """Whether the plain computation would take more than some seconds."""
    nb = 3 ** dim - 1
    kept = steps > 1 and cells * nb * 8 <= 60 << 30
    return cells * nb * (3 * r + steps if kept else 3 * r * steps) > 2.2e12


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch":
        mix, cells, first, state = _batch_states(case, seed)
        if sum(cells) * case["steps"] > 2e10:
            return None
        for (fam, r, _), c, o in zip(mix, cells, first):
            v = state[int(o):int(o) + c]
            v.copy_(_Plain(fam, r).step(v, case["steps"], W.LIFE_B3S23))
        return state
    fam, r = W.FAMILIES[case["family"]], case["r"]
    plain = _Plain(fam, r)
    if kind == "maps":
        omega, coords = _points(case, seed)
        return {"coords": plain.lam(omega), "omega": plain.nu(coords), "compact": plain.compact(coords)}
    cells = fam.k ** r
    if _too_long(cells, r, case["steps"], fam.dim):
        return None
    out = plain.step(_bernoulli(cells, case["p"], _generator(seed)), case["steps"], RULES[case["rule"]])
    if kind == "host":
        return out.cpu()
    if kind == "box":
        box = torch.zeros((fam.s ** r) ** fam.dim, dtype=torch.uint8, device="cuda")
        for lo in range(0, cells, 1 << 25):
            c = plain.lam(torch.arange(lo, min(lo + (1 << 25), cells), dtype=torch.int64, device="cuda"))
            box[sum(c[:, a] * plain.side ** a for a in range(fam.dim))] = out[lo:lo + (1 << 25)]
        return {"box": box, "compact": out}
    return out
