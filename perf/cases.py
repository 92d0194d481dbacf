"""What a user of this framework has it do, as cases that can be timed and whose outputs can be compared.

A case is a dict of plain values.  Its "kind" says which public calls one pass makes:

  run       System.step(steps), then the new frame (positions, velocities, forces) into pinned host buffers
  batch     Batch.step(steps) of several resident systems, then every system's frame
  turnover  one request of a server: Batch.try_add, step(steps) of all residents, get_state, remove
  resume    a System's checkpoint restored from pinned host memory, step(steps), the new checkpoint back
  analysis  step(steps) with running means, then observables() and the pair-distance histogram
  cells     cells_noalloc on positions that are in device memory already

The remaining values are the box edges, the density, the precision (32 or 64 bits), the chains in the
fluid, the bead types and the noise.
"""
import math

import numpy as np
import torch

from paper_1804_06205_gb300 import dpd

KT, LAM = 1.0, 0.65
HARMONIC, MORSE_PAPER, MORSE = 1, 2, 3


def _case(kind, edges, steps, bits=32, chains="none", types=1, rho=3.0, noise=0, **more):
    lx, ly, lz = edges if isinstance(edges, tuple) else (edges,) * 3
    return dict(kind=kind, lx=lx, ly=ly, lz=lz, rho=rho, bits=bits, chains=chains, types=types,
                noise=noise, steps=steps, **more)


def listed():
    """The cases that stand for the framework's use."""
    edge_100k = round((100_000 / 3.0) ** (1.0 / 3.0), 6)
    return [
        # the smallest fluid that the tests and the paper's benchmark fluid use: launches and latency count
        dict(_case("run", 10.0, 20), name="fluid_3k"),
        # the paper's protein model: one bonded chain in 24,000 beads, run for thousands of steps
        dict(_case("run", 20.0, 20, chains="helix", types=2), name="helix_24k"),
        # the largest row of the paper's timing table: an edge that is no whole number of cells
        dict(_case("run", edge_100k, 20), name="table_100k"),
        # a polymer melt: every bead in a bonded chain
        dict(_case("run", 32.0, 20, chains="melt", types=2), name="melt_98k"),
        # the headline fluid, far above the L2 cache
        dict(_case("run", 100.0, 10, types=2), name="fluid_3m"),
        # peptide-like chains in solvent on the FP64 path
        dict(_case("run", 40.0, 10, bits=64, chains="peptide", types=2), name="peptide_192k_f64"),
        # the headline fluid's recipe on the FP64 path, above the L2 cache
        dict(_case("run", 70.0, 4, bits=64, types=2), name="fluid_1m_f64"),
        # what a server holds at the stream's arrival rate: a few uneven systems, edges 8 to 24
        dict(_case("batch", 8.0, 20, chains="tenth", types=2, systems=9, edge_max=24.0), name="serving_9"),
        # one request of a server with other systems resident: admission, a chunk of steps, read-back, removal
        dict(_case("turnover", 8.0, 20, chains="tenth", types=2, systems=6, edge_max=20.0), name="turnover_6"),
        # a state kept on the host: restored, advanced and read back each time
        dict(_case("resume", 70.0, 1, types=2), name="resume_1m"),
        # statistics of a run: running means, observables, g(r)
        dict(_case("analysis", 32.0, 20, chains="tenth", types=2, rmax=3.0, bins=60), name="analysis_98k"),
        # the cell division alone, for a caller that owns its device memory
        dict(_case("cells", 70.0, 0), name="cells_1m"),
    ]


def _log_uniform(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _edges(rng, n, rho):
    """A box, not a cube in general, that holds about n beads."""
    if rng.random() < 0.3:
        e = max(3.0, round((n / rho) ** (1.0 / 3.0), 3))
        return e, e, e
    r = [rng.uniform(0.6, 1.7) for _ in range(3)]
    s = (n / rho / (r[0] * r[1] * r[2])) ** (1.0 / 3.0)
    e = [max(3.0, round(x * s, 3)) for x in r]
    if rng.random() < 0.3:
        e = [float(max(3, round(x))) for x in e]
    return tuple(e)


def draw(rng):
    """One more case of the ranges that the listed ones stand for."""
    kind = rng.choice(["run"] * 9 + ["batch"] * 2 + ["turnover", "resume", "analysis", "cells"])
    noise = 1 if rng.random() < 0.15 else 0
    types = rng.choice([1, 2, 2, 3])
    if kind in ("batch", "turnover"):
        count = rng.randint(2, 12 if kind == "batch" else 7)
        lo, hi = rng.uniform(6.0, 12.0), rng.uniform(13.0, 24.0)
        return _case(kind, round(lo, 3), rng.randint(10, 25), bits=rng.choice([32, 32, 64]), chains="tenth",
                     types=rng.choice([1, 2]), noise=noise, systems=count, edge_max=round(hi, 3))
    if kind == "resume":
        return _case(kind, _edges(rng, _log_uniform(rng, 20_000, 1_500_000), 3.0), rng.randint(1, 2),
                     bits=rng.choice([32, 32, 64]), types=types, noise=noise)
    if kind == "analysis":
        e = _edges(rng, _log_uniform(rng, 6_000, 90_000), 3.0)
        e = tuple(max(8.0, x) for x in e)
        return _case(kind, e, rng.randint(10, 20), bits=rng.choice([32, 64]), types=types, noise=noise,
                     chains=rng.choice(["none", "tenth"]), rmax=rng.choice([2.0, 2.5, 3.0]),
                     bins=rng.choice([50, 60, 100]))
    if kind == "cells":
        return _case(kind, _edges(rng, _log_uniform(rng, 5_000, 2_000_000), 3.0), 0)
    bits = rng.choice([32, 32, 64])
    rho = rng.choice([3.0, 3.0, 3.0, 4.0])
    n = _log_uniform(rng, 800, (2_400_000 if bits == 32 else 800_000) / (rho / 3.0) ** 2)
    chains = rng.choice(["none", "none", "tenth", "melt", "peptide", "helix"])
    if chains == "helix":
        n, types = min(n, 120_000), 2
    steps = rng.randint(8, 22) if n < 300_000 else rng.randint(3, 8 if bits == 32 else 4)
    return _case("run", _edges(rng, max(n, 300), rho), steps, bits=bits, chains=chains, types=types, rho=rho,
                 noise=noise)


# ---- inputs -------------------------------------------------------------------------------------


def _walks(rng, count, length, step, box):
    """Chains as random walks of a fixed step from uniform starts, wrapped into the box."""
    d = rng.normal(size=(count, length - 1, 3))
    d *= step / np.linalg.norm(d, axis=2, keepdims=True)
    w = np.concatenate([np.zeros((count, 1, 3)), np.cumsum(d, axis=1)], axis=1)
    return np.mod((w + rng.random((count, 1, 3)) * box).reshape(-1, 3), box)


def _links(count, length, apart, kind, r0, k, alpha=0.0):
    i = (np.arange(count)[:, None] * length + np.arange(length - apart)[None, :]).ravel()
    m = i.size
    return dict(i=i.astype(np.int32), j=(i + apart).astype(np.int32), kind=np.full(m, kind, np.int32),
                r0=np.full(m, r0), k=np.full(m, k), alpha=np.full(m, alpha))


def _system(c, seed):
    """One system's box, parameters, bonds and initial state, from the seed alone."""
    rng = np.random.default_rng(seed)
    box = np.array([c["lx"], c["ly"], c["lz"]])
    n = max(1, int(round(c["rho"] * float(np.prod(box)))))
    nt, chains = c["types"], c["chains"]
    a = np.full((nt, nt), 25.0 if nt == 1 else float(rng.uniform(28.0, 45.0)))
    np.fill_diagonal(a, 25.0)
    gamma, dt, parts = 4.5, 0.04, []
    count, length, step = {"none": (0, 10, 0.5), "melt": (n // 10, 10, 0.5), "tenth": (n // 100, 10, 0.5),
                           "peptide": (n // 960, 20, 0.5), "helix": (1 if n >= 60 else 0, 60, 0.6)}[chains]
    if count and chains in ("melt", "tenth"):
        parts = [_links(count, length, 1, HARMONIC, 0.0, 4.0)]
    elif count and chains == "peptide":
        parts = [_links(count, length, 1, HARMONIC, 0.5, 4.0), _links(count, length, 2, MORSE, 0.7, 5.0, 3.0),
                 _links(count, length, 4, MORSE, 1.0, 5.0, 3.0)]
        dt = 0.02  # as in the protein model: random chains start far from the Morse terms' minima
    elif count:
        parts = [_links(1, 60, 1, HARMONIC, 0.6, 160.0), _links(1, 60, 2, HARMONIC, 1.2, 80.0),
                 _links(1, 60, 2, MORSE_PAPER, 0.9, 12.0, 8.0), _links(1, 60, 4, MORSE_PAPER, 0.6, 12.0, 8.0)]
        gamma, dt = 4.2, 0.02
        a = np.full((nt, nt), 55.0)
        np.fill_diagonal(a, 50.0)
    bonds = {k: np.concatenate([p[k] for p in parts]) for k in parts[0]} if parts else None
    m = count * length
    pos = rng.random((n, 3)) * box
    if m:
        pos[:m] = _walks(rng, count, length, step, box)
    pos = np.where(pos >= box, 0.0, pos)
    types = rng.integers(0, nt, n).astype(np.int32)
    if chains == "melt":
        types[:m] = (np.arange(m) % 10 >= 5) if nt > 1 else 0
    elif chains in ("peptide", "helix"):
        types[:m], types[m:] = 0, nt - 1
    vel = rng.standard_normal((n, 3)) * math.sqrt(KT)
    vel -= vel.mean(axis=0, keepdims=True)
    return dict(box=box, n=n, types=types, a=a, gamma=gamma, dt=dt, bonds=bonds, pos=pos, vel=vel,
                seed=(seed * 7919 + 11) & 0xFFFFFFFFFFFF, noise=c["noise"])


def _systems(c, seed):
    """The systems of a batch, edges from lx to edge_max in even steps."""
    m = c["systems"]
    out = []
    for k in range(m):
        e = c["lx"] + (c["edge_max"] - c["lx"]) * (k / max(1, m - 1))
        out.append(_system(dict(c, lx=e, ly=e, lz=e), seed * 1000 + k))
    return out


def _create(c, s, **opt):
    return dpd.System(s["box"], s["types"], s["a"], s["gamma"], KT, s["dt"], bonds=s["bonds"], lam=LAM,
                      seed=s["seed"], noise=s["noise"],
                      precision=dpd.DPD_FP64 if c["bits"] == 64 else dpd.DPD_FP32, **opt)


def _admit(b, s):
    return b.try_add(s["box"], s["types"], s["a"], s["gamma"], KT, s["dt"], s["pos"], s["vel"],
                     bonds=s["bonds"], lam=LAM, seed=s["seed"])


def prepare(case, seed):
    """The plan that a program keeps (a System, a Batch, buffers) with its initial state set."""
    c = case
    if c["kind"] in ("batch", "turnover"):
        sys = _systems(c, seed)
        room = [int(np.prod(np.floor(s["box"]))) for s in sys]
        links = sum(len(s["bonds"]["i"]) for s in sys if s["bonds"] is not None)
        b = dpd.Batch(sum(s["n"] for s in sys), sum(room), max(1, links), max_systems=len(sys), noise=c["noise"],
                      precision=dpd.DPD_FP64 if c["bits"] == 64 else dpd.DPD_FP32)
        new = sys[len(sys) // 2] if c["kind"] == "turnover" else None
        ids = [_admit(b, s) for s in sys if s is not new]
        return dict(case=c, batch=b, ids=ids, new=new)
    if c["kind"] == "cells":
        rng = np.random.default_rng(seed)
        box = np.array([c["lx"], c["ly"], c["lz"]])
        n = max(1, int(round(c["rho"] * float(np.prod(box)))))
        # a few beads lie outside the box, as after a move that was not wrapped yet
        pos = torch.from_numpy((rng.random((n, 3)) * 1.01 - 0.005) * box).cuda()
        i32 = dict(dtype=torch.int32, device="cuda")
        return dict(case=c, box=box, n=n, pos=pos, key=torch.empty(n, **i32), order=torch.empty(n, **i32),
                    start=torch.empty(int(np.prod(np.floor(box))) + 1, **i32))
    s = _system(c, seed)
    h = _create(c, s, sample_every=5 if c["kind"] == "analysis" else 0)
    h.set_state(s["pos"], s["vel"], 0)
    st = dict(case=c, system=h)
    if c["kind"] == "run":
        st["frame"] = [torch.empty((s["n"], 3), dtype=torch.float64, pin_memory=True) for _ in range(3)]
    if c["kind"] == "resume":
        nb = h.checkpoint_bytes()
        st["kept"], st["next"] = (torch.empty(nb, dtype=torch.uint8, pin_memory=True) for _ in range(2))
        h.get_checkpoint_ptr(st["kept"].data_ptr(), nb)
    return st


# ---- one pass -----------------------------------------------------------------------------------


def run(state):
    c = state["case"]
    if c["kind"] == "run":
        p, v, f = state["frame"]
        state["system"].step(c["steps"])
        state["system"].get_state_ptr(p.data_ptr(), v.data_ptr(), f.data_ptr())
        return {"pos": p, "vel": v, "force": f}
    if c["kind"] == "batch":
        b = state["batch"]
        b.step(c["steps"])
        return [dict(zip(("pos", "vel", "force"), b.get_state(i)[:3])) for i in state["ids"]]
    if c["kind"] == "turnover":
        b = state["batch"]
        i = _admit(b, state["new"])
        b.step(c["steps"])
        done = b.get_state(i)
        b.remove(i)
        return dict(zip(("pos", "vel", "force"), done[:3]))
    if c["kind"] == "resume":
        h, a, z = state["system"], state["kept"], state["next"]
        h.set_checkpoint_ptr(a.data_ptr(), a.numel())
        h.step(c["steps"])
        h.get_checkpoint_ptr(z.data_ptr(), z.numel())
        return {"checkpoint": z}
    if c["kind"] == "analysis":
        h = state["system"]
        h.step(c["steps"])
        seen = h.observables()
        return {"observables": seen, "pairs": h.gr_counts(c["rmax"], c["bins"]).astype(np.int64)}
    dpd.cells_noalloc(state["pos"].data_ptr(), state["n"], state["box"], state["key"].data_ptr(),
                      state["order"].data_ptr(), state["start"].data_ptr(),
                      torch.cuda.current_stream().cuda_stream or None)
    return {"key": state["key"], "order": state["order"], "cell_start": state["start"]}


def _beads(c):
    if c["kind"] in ("batch", "turnover"):
        m = c["systems"]
        return sum(round(c["rho"] * (c["lx"] + (c["edge_max"] - c["lx"]) * (k / max(1, m - 1))) ** 3)
                   for k in range(m))
    return round(c["rho"] * c["lx"] * c["ly"] * c["lz"])


def work(case):
    """Each step reads and writes r, v and f (a state this framework serves does not stay on the chip), tests
    the unique candidates of the 27 cells (8 operations) and evaluates the unique pairs (150 operations)."""
    c, n = case, _beads(case)
    word, rho = c["bits"] // 8, c["rho"]
    if c["kind"] == "cells":
        cells = math.floor(c["lx"]) * math.floor(c["ly"]) * math.floor(c["lz"])
        return {"bytes": n * (24 + 4 + 4) + 4 * cells, "flops": n * 30}
    bytes_, flops = c["steps"] * n * 18 * word, c["steps"] * n * (13.5 * rho * 8 + 2.0944 * rho * 150)
    if c["kind"] == "resume":
        bytes_ += 2 * n * (40 if word == 4 else 72)
    elif c["kind"] == "analysis":
        flops += n * 13 * (4.1888 * c["rmax"] ** 3 * rho / 2)
    else:
        bytes_ += n * 72
    return {"bytes": bytes_, "flops": flops}


# ---- the same numbers in plain 64-bit torch ------------------------------------------------------


def _mul32(a, b):
    """High and low halves of the 64-bit product of 32-bit words, in int64."""
    lo, hi = (a & 0xFFFF) * b, (a >> 16) * b
    mid = hi + (lo >> 16)
    return mid >> 16, ((mid & 0xFFFF) << 16) | (lo & 0xFFFF)


def _theta(i, j, step, seed, noise):
    """The pair's noise: Philox4x32-10 of (min id, max id, step), then Box-Muller (or a scaled uniform)."""
    c0, c1 = torch.minimum(i, j), torch.maximum(i, j)
    c2 = torch.full_like(c0, step & 0xFFFFFFFF)
    c3 = torch.full_like(c0, step >> 32)
    k0, k1 = seed & 0xFFFFFFFF, seed >> 32
    for _ in range(10):
        h0, l0 = _mul32(c0, 0xD2511F53)
        h1, l1 = _mul32(c2, 0xCD9E8D57)
        c0, c1, c2, c3 = h1 ^ c1 ^ k0, l1, h0 ^ c3 ^ k1, l0
        k0, k1 = (k0 + 0x9E3779B9) & 0xFFFFFFFF, (k1 + 0xBB67AE85) & 0xFFFFFFFF
    u0, u1 = ((2 * (x >> 9) + 1).double() * 2.0 ** -24 for x in (c0, c1))
    if noise:
        return math.sqrt(3.0) * (2.0 * u0 - 1.0)
    return torch.sqrt(-2.0 * torch.log(u0)) * torch.cos(2.0 * math.pi * u1)


class _Exact:
    """One system in 64 bits: the paper's equations, with cells only to find the pairs."""

    def __init__(self, s):
        dev = "cuda" if torch.cuda.is_available() else "cpu"
        t = lambda x: torch.from_numpy(np.ascontiguousarray(x)).to(dev)  # noqa: E731
        self.s, self.L = s, t(s["box"])
        self.nc = [int(x) for x in np.floor(s["box"])]
        self.types, self.a = t(s["types"]).long(), t(s["a"])
        self.sig = math.sqrt(2.0 * s["gamma"] * KT) / math.sqrt(s["dt"])
        self.bonds = None if s["bonds"] is None else {k: t(v) for k, v in s["bonds"].items()}
        self.r, self.v, self.step = t(s["pos"]), t(s["vel"]), 0
        self.f = self.forces(self.v)

    def image(self, d):
        return d - self.L * torch.round(d / self.L)

    def pairs(self):
        """The unique pairs closer than 1, as (i, j)."""
        nx, ny, nz = self.nc
        n = torch.tensor(self.nc, device=self.r.device)
        c = torch.minimum((self.r * (n / self.L)).floor().long(), n - 1)
        key = (c[:, 2] * ny + c[:, 1]) * nx + c[:, 0]
        order = torch.argsort(key, stable=True)
        count = torch.bincount(key, minlength=nx * ny * nz)
        first = torch.cumsum(count, 0) - count
        slot = torch.arange(len(order), device=order.device) - first[key[order]]
        table = torch.full((nx * ny * nz, int(count.max())), -1, device=order.device)
        table[key[order], slot] = order
        got = []
        me = torch.arange(len(order), device=order.device)[:, None]
        for dz, dy, dx in [(z, y, x) for z in (-1, 0, 1) for y in (-1, 0, 1) for x in (-1, 0, 1)]:
            if (dz, dy, dx) < (0, 0, 0):
                continue
            near = (((c[:, 2] + dz) % nz) * ny + (c[:, 1] + dy) % ny) * nx + (c[:, 0] + dx) % nx
            j = table[near]
            ok = (j >= 0) & ((j > me) if (dz, dy, dx) == (0, 0, 0) else True)
            d = self.image(self.r[:, None, :] - self.r[j.clamp(min=0)])
            i, k = torch.nonzero(ok & (d.square().sum(2) < 1.0), as_tuple=True)
            got.append(torch.stack([i, j[i, k]]))
        return torch.cat(got, 1)

    def forces(self, v):
        s = self.s
        i, j = self.pairs()
        d = self.image(self.r[i] - self.r[j])
        r = d.square().sum(1).sqrt()
        e = torch.where(r[:, None] > 0, d / r[:, None], torch.zeros_like(d))
        w, a = 1.0 - r, self.a[self.types[i], self.types[j]]
        th = _theta(i, j, self.step, s["seed"], s["noise"])
        mag = a * w - s["gamma"] * w * w * (e * (v[i] - v[j])).sum(1) + self.sig * w * th
        f = torch.zeros_like(self.r)
        f.index_add_(0, i, mag[:, None] * e)
        f.index_add_(0, j, -mag[:, None] * e)
        self.pair_sums = (float((r * a * w).sum()), float((0.5 * a * w * w).sum()))
        self.bond_sums = (0.0, 0.0)
        if self.bonds is not None:
            b = self.bonds
            i, j, kind, r0, k, al = b["i"].long(), b["j"].long(), b["kind"], b["r0"], b["k"], b["alpha"]
            d = self.image(self.r[i] - self.r[j])
            r = d.square().sum(1).sqrt()
            x = r - r0
            ep, em = torch.exp(-al * x.abs()), torch.exp(-al * x)
            pull = torch.where(kind == HARMONIC, k * x, torch.where(
                kind == MORSE_PAPER, 2 * k * al * ep * (1 - ep), 2 * k * al * em * (1 - em)))
            u = torch.where(kind == HARMONIC, 0.5 * k * x * x, torch.where(
                kind == MORSE_PAPER, k * (1 - ep) ** 2, k * ((1 - em) ** 2 - 1)))
            fb = torch.where(r[:, None] > 0, -pull[:, None] * d / r[:, None], torch.zeros_like(d))
            f.index_add_(0, i, fb)
            f.index_add_(0, j, -fb)
            self.bond_sums = (float((d * fb).sum()), float(u.sum()))
        return f

    def advance(self, steps, each=None):
        dt = self.s["dt"]
        for _ in range(steps):
            r = self.r + dt * self.v + 0.5 * dt * dt * self.f
            self.r = r - self.L * torch.floor(r / self.L)
            self.r = torch.where(self.r >= self.L, self.r - self.L, self.r)
            self.step += 1
            f = self.forces(self.v + LAM * dt * self.f)
            self.v = self.v + 0.5 * dt * (self.f + f)
            self.f = f
            if each is not None:
                each()

    def frame(self):
        return {"pos": self.r, "vel": self.v, "force": self.f}

    def means(self):
        """kT and the pressure with its parts."""
        v2, vol = float(self.v.square().sum()), float(self.L.prod())
        p = [x / (3.0 * vol) for x in (v2, self.pair_sums[0], self.bond_sums[0])]
        return dict(sum_v2=v2, kT=v2 / (3.0 * len(self.v) - 3.0) if len(self.v) > 1 else 0.0, p_ideal=p[0],
                    p_cons=p[1], p_bond=p[2], p_total=sum(p), e_pair=self.pair_sums[1], e_bond=self.bond_sums[1])


def exact(case, seed):
    c = case
    if c["kind"] in ("resume", "cells"):
        return None  # bytes and whole numbers
    if c["kind"] == "batch":
        out = []
        for s in _systems(c, seed):
            x = _Exact(s)
            x.advance(c["steps"])
            out.append(x.frame())
        return out
    if c["kind"] == "turnover":
        x = _Exact(_systems(c, seed)[c["systems"] // 2])
        x.advance(c["steps"])
        return x.frame()
    x = _Exact(_system(c, seed))
    if c["kind"] == "run":
        x.advance(c["steps"])
        return x.frame()
    seen = []
    x.advance(c["steps"], lambda: seen.append(x.means()) if x.step % 5 == 0 else None)
    k = len(seen)
    # the total momentum is zero but for rounding, and the histogram holds whole numbers
    return {"observables": dict(x.means(), momentum=None, step=None, status=None, n_samples=None,
                                kT_mean=sum(m["kT"] for m in seen) / k if k else 0.0,
                                p_mean=sum(m["p_total"] for m in seen) / k if k else 0.0), "pairs": None}
