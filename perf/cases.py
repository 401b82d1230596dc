"""Performance cases of the level-set grain-growth library.

A case is a simulation as a user's program runs it through the public binding
(``paper_1701_06658_gb300.lsgg``): a microstructure is created from host
arrays (seed points, weights, orientations, energies or a label field), it is
advanced, its grain volumes are read at intervals and its voxel owner map (on
request its boxes and functions, a restart file's content) at the end, and it
is closed.  A serving case submits independent simulations to one server and
waits for all of them.

``prepare`` holds what such a program has in hand before the call: the host
arrays, the pinned or device buffers the results land in, a running server.
Every number comes from the seed.  ``exact`` is the same simulation in plain
torch in 64 bits: grain functions in windows around their boxes, one step at
a time (heat-kernel convolution, comparison with the largest other function,
taxicab re-initialisation, box update), without the library.
"""
import math

import numpy as np
import torch

from paper_1701_06658_gb300 import inputs as I
from paper_1701_06658_gb300 import lsgg as L

EPS, HALO, RADIUS, DT = 7.0, 5, 5, 1.0
CELLS_PER_GRAIN = 3355.0          # the 256^3 / 5000 workload's density, also the served requests' one
ENERGY_SCALE = 4.07e-3            # magnetic energy density at cos^2 = 1, grid units
THETA_MAX, MOB_LOW = 15.0, 0.1    # Read-Shockley law and low-angle mobility
SERVE_SEED = 1000                 # draws the served requests' sizes and step counts


# ---------------------------------------------------------------- the cases

def _sim(name, nx, ny, nz, grains, steps, every, start="voronoi", physics="ideal", bf16=False, state=False,
         device=False, cols=0):
    """Advance ``steps`` steps, reading the volumes every ``every``; ``state``: boxes and functions at the end
    too; ``device``: the owner map into device memory instead of a pinned host buffer; ``cols``: grains per row
    of the "hex" start's lattice."""
    return {"name": name, "kind": "sim", "nx": nx, "ny": ny, "nz": nz, "grains": grains, "steps": steps,
            "every": every, "start": start, "physics": physics, "bf16": bf16, "state": state, "device": device,
            "cols": cols}


def listed():
    return [
        # the smallest served domain (32^3, 20 grains): the boxes meet the domain's periodic edges, a step is
        # launches and latency; ends with a restart file
        _sim("small_32", 32, 32, 32, 20, 60, 10, state=True),
        # the accuracy configuration (64^3, 50 grains, 20 steps) with volumes after every step
        _sim("accuracy_64", 64, 64, 64, 50, 20, 1, state=True),
        # a voxelised measurement: a label field on an odd, non-cubic domain
        _sim("labels_ragged", 149, 97, 61, 263, 30, 5, start="labels"),
        # 2D growth (von Neumann-Mullins studies): hexagon-like grains of about 20 cells across
        _sim("plane_512", 512, 512, 1, 26 * 26, 60, 10, start="hex", cols=26),
        # the headline workload: 256^3, 5000 Voronoi grains, ideal growth
        _sim("ideal_256", 256, 256, 256, 5000, 100, 10),
        # the reduced-storage variant on a mid-size odd domain
        _sim("bf16_191", 191, 191, 191, 2077, 50, 5, bf16=True),
        # non-ideal growth at the size of a parameter study: lognormal grains, Read-Shockley boundaries
        _sim("read_shockley_160", 160, 160, 160, 1221, 60, 10, start="laguerre", physics="read_shockley"),
        # the same at full size (512^3, 40 000 grains): the largest arenas
        _sim("read_shockley_512", 512, 512, 512, 40000, 24, 8, start="laguerre", physics="read_shockley", device=True),
        # magnetically driven growth at full size (384^3, 10 000 grains)
        _sim("magnetic_384", 384, 384, 384, 10000, 30, 10, physics="magnetic", device=True),
        # serving: independent simulations of 32^3 to 128^3, all submitted at once
        {"name": "serve_24", "kind": "serve", "count": 24, "lo": 32, "hi": 128, "steps_hi": 80},
    ]


def draw(rng):
    def log_between(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["ideal", "ideal", "ideal", "labels", "hex", "read_shockley", "magnetic", "serve"])
    if kind == "serve":
        return {"kind": "serve", "count": rng.randint(8, 32), "lo": rng.choice([32, 48]),
                "hi": rng.choice([64, 96, 112, 128]), "steps_hi": rng.randint(30, 80)}
    steps = rng.randint(10, 50)
    every = rng.randint(1, 10)
    if kind == "hex":
        nx, ny = log_between(128, 768), log_between(128, 768)
        cols, rows = max(2, nx // 20), max(2, 2 * (ny // 40))
        c = _sim("", nx, ny, 1, cols * rows, steps, every, start="hex", cols=cols)
    else:
        n = log_between(32, 256 if kind == "ideal" else 192)
        dims = [n, n, n] if rng.random() < 0.4 else [max(24, int(n * rng.uniform(0.6, 1.3))) for _ in range(3)]
        per_grain = rng.uniform(2400.0, 5300.0)
        grains = max(8, int(round(dims[0] * dims[1] * dims[2] / per_grain)))
        c = _sim("", *dims, grains, steps, every,
                 start={"labels": "labels", "read_shockley": "laguerre"}.get(kind, "voronoi"),
                 physics=kind if kind in ("read_shockley", "magnetic") else "ideal",
                 bf16=kind == "ideal" and rng.random() < 0.3, state=n < 72)
    del c["name"]
    return c


# ---------------------------------------------------------------- inputs

def _requests(case):
    """(side, grains, steps) of the served requests: the same for every seed."""
    reqs = I.serving_requests(case["count"], 1.0, SERVE_SEED, sizes=tuple(range(case["lo"], case["hi"] + 1, 16)),
                              steps_range=(10, case["steps_hi"]))
    return [(r.n, r.n_grains, r.steps) for r in reqs]


def _power_labels(seeds, weights, dims):
    """(nz, ny, nx) labels of the periodic power diagram in 64 bits, lowest id on ties: per block of cells only
    the seeds that can be nearest to one of them."""
    nx, ny, nz = dims
    n = torch.tensor([nx, ny, nz], dtype=torch.float64, device="cuda")
    s = torch.as_tensor(seeds, dtype=torch.float64, device="cuda")
    w = torch.zeros(len(s), dtype=torch.float64, device="cuda") if weights is None else \
        torch.as_tensor(weights, dtype=torch.float64, device="cuda")
    out = torch.empty((nz, ny, nx), dtype=torch.int64, device="cuda")
    B = 32
    for z0 in range(0, nz, B):
        for y0 in range(0, ny, B):
            for x0 in range(0, nx, B):
                hi = (min(x0 + B, nx) - 1, min(y0 + B, ny) - 1, min(z0 + B, nz) - 1)
                half = torch.tensor([(h - l) / 2 for h, l in zip(hi, (x0, y0, z0))], dtype=torch.float64, device="cuda")
                mid = torch.tensor([(h + l) / 2 for h, l in zip(hi, (x0, y0, z0))], dtype=torch.float64, device="cuda")
                d = (s - mid).remainder(n)
                d = torch.minimum(d, n - d)
                near = ((d - half).clamp_min(0) ** 2).sum(1) - w
                far = (torch.minimum(d + half, n / 2) ** 2).sum(1) - w
                cand = torch.nonzero(near <= far.min() + 1e-6).flatten()
                ax = [torch.arange(l, h + 1, dtype=torch.float64, device="cuda") for l, h in zip((x0, y0, z0), hi)]
                r = []
                for a in range(3):
                    e = ax[a][:, None] - s[cand, a][None, :]
                    r.append((e - n[a] * torch.round(e / n[a])) ** 2)
                p = (r[0][None, None] + r[1][None, :, None]) + r[2][:, None, None] - w[cand]
                out[z0:hi[2] + 1, y0:hi[1] + 1, x0:hi[0] + 1] = cand[p.argmin(-1)]
    return out


def _arrays(case, seed):
    """The host arrays a simulation starts from."""
    dims = (case["nx"], case["ny"], case["nz"])
    g = case["grains"]
    a = {}
    if case["start"] == "hex":
        a["seeds"] = I.jittered_hex_seeds(seed, dims[0], dims[1], case["cols"], g // case["cols"])
    else:
        a["seeds"] = I.voronoi_seeds(seed, g, dims)
    if case["start"] == "laguerre":
        a["weights"] = I.laguerre_weights(seed, g, dims)
    if case["physics"] == "read_shockley":
        a["quats"] = I.random_quaternions(seed, g)
    if case["physics"] == "magnetic":
        q = I.random_quaternions(seed, g)
        axis = np.stack([2 * (q[:, 1] * q[:, 3] + q[:, 0] * q[:, 2]), 2 * (q[:, 2] * q[:, 3] - q[:, 0] * q[:, 1]),
                         1 - 2 * (q[:, 1] ** 2 + q[:, 2] ** 2)], axis=1)
        f = np.array([0.0, math.cos(math.radians(32.0)), math.sin(math.radians(32.0))])
        a["energy"] = ENERGY_SCALE * (axis @ f) ** 2
    if case["start"] == "labels":
        a = {"labels": _power_labels(a["seeds"], None, dims).to(torch.int32).cpu().numpy()}
    return a


def _pinned(shape, dtype):
    return torch.empty(shape, dtype=dtype, pin_memory=True)


def _phi_room(case):
    """Values of the buffer a restart file's functions land in (packed; the rest stays zero)."""
    return 2 * int(_box_cells(case["nx"], case["ny"], case["nz"], case["grains"]))


def prepare(case, seed):
    if case["kind"] == "serve":
        reqs = _requests(case)
        seeds = [I.voronoi_seeds(1009 * seed + k, g, (n, n, n)) for k, (n, g, _) in enumerate(reqs)]
        return {"case": case, "reqs": reqs, "seeds": seeds, "server": L.Server(150_000_000_000),
                "volumes": np.zeros(sum(g for _, g, _ in reqs))}
    shape = (case["nz"], case["ny"], case["nx"])
    reads = -(-case["steps"] // case["every"])
    kw = {"physics": {"ideal": L.PHYSICS_IDEAL, "read_shockley": L.PHYSICS_READ_SHOCKLEY,
                      "magnetic": L.PHYSICS_MAGNETIC}[case["physics"]],
          "storage": L.STORAGE_BF16 if case["bf16"] else L.STORAGE_FP32, **_arrays(case, seed)}
    owner = torch.empty(shape, dtype=torch.int32, device="cuda") if case["device"] else _pinned(shape, torch.int32)
    state = {"case": case, "kw": kw, "volumes": _pinned((reads, case["grains"]), torch.float64), "owner": owner}
    if case["state"]:
        state["phi"] = np.zeros(_phi_room(case), np.float32)
    return state


# ---------------------------------------------------------------- one pass

def run(state):
    case = state["case"]
    if case["kind"] == "serve":
        server, at = state["server"], 0
        tickets = [server.submit(n, n, n, g, steps, DT, seeds=s)
                   for (n, g, steps), s in zip(state["reqs"], state["seeds"])]
        for t, (_, g, _) in zip(tickets, state["reqs"]):
            server.wait(t)
            state["volumes"][at:at + g] = server.volumes(t)
            server.release(t)
            at += g
        return {"volumes": state["volumes"]}
    out = {"volumes": state["volumes"], "owner": state["owner"]}
    volumes = state["volumes"].numpy()
    with L.Microstructure(case["nx"], case["ny"], case["nz"], case["grains"], **state["kw"]) as ms:
        done = 0
        for row in volumes:
            n = min(case["every"], case["steps"] - done)
            ms.step(n, DT)
            ms.grain_volumes(row)
            done += n
        if case["device"]:
            L.voxel_owner_device(ms.ctx, state["owner"].data_ptr(), state["owner"].numel())
            ms.sync()
        else:
            ms.voxel_owner(state["owner"].numpy())
        if case["state"]:
            phi = L.get_phi(ms.ctx)
            state["phi"][:phi.size] = phi
            out["boxes"], out["phi"] = ms.boxes(), state["phi"]
    return out


# ---------------------------------------------------------------- the work of a pass

def _box_cells(nx, ny, nz, grains):
    """Cells of the grains' boxes: a cell of the tessellation reaches about 1.36 of its mean diameter per axis
    (1.25 in 2D), plus the halo."""
    dim = 2 if nz == 1 else 3
    d = (nx * ny * nz / grains) ** (1.0 / dim) * (1.36 if dim == 3 else 1.25) + 2 * HALO
    return grains * min(d, nx) * min(d, ny) * (min(d, nz) if dim == 3 else 1)


def work(case):
    sims = [(n, n, n, g, s, 4, False) for n, g, s in _requests(case)] if case["kind"] == "serve" else \
        [(case["nx"], case["ny"], case["nz"], case["grains"], case["steps"], 2 if case["bf16"] else 4,
          case["physics"] != "ideal")]
    bytes_, flops = 0.0, 0.0
    for nx, ny, nz, g, steps, width, ids in sims:
        cells = _box_cells(nx, ny, nz, g)
        # a step reads and writes every box cell's state once (with pair physics its neighbour id too); its taps
        # are an FMA each per axis, about 14 operations more for comparison and re-initialisation
        bytes_ += steps * cells * 2 * (width + (4 if ids else 0)) + 4 * nx * ny * nz + 24 * g
        flops += steps * cells * (2 * (2 * RADIUS + 1) * (2 if nz == 1 else 3) + 14)
    return {"bytes": bytes_, "flops": flops}


# ---------------------------------------------------------------- 64-bit reference

class _Exact:
    """All grains' functions in windows (G, wz, wy, wx) at their boxes' origins, -EPS beyond a box."""

    def __init__(self, dims, g):
        self.N = (dims[2], dims[1], dims[0])
        self.axes = (1, 2) if dims[2] == 1 else (0, 1, 2)
        self.G = g
        k = torch.arange(-RADIUS, RADIUS + 1, dtype=torch.float64)
        t = torch.exp(-k * k / (4.0 * DT))
        self.taps = (t / t.sum()).tolist()

    # box helpers: o, n are (G, 3) origins and dims in (z, y, x) order
    def layout(self, o, n):
        self.o, self.n = o, n
        self.w = [int(n[:, a].max()) for a in range(3)]
        self.full = [n[:, a] == self.N[a] for a in range(3)]
        self.at, inside = [], []
        for a in range(3):
            l = torch.arange(self.w[a], device="cuda")
            self.at.append((o[:, a, None] + l) % self.N[a])
            inside.append(l < n[:, a, None])
        self.inside = inside[0][:, :, None, None] & inside[1][:, None, :, None] & inside[2][:, None, None, :]
        self.cell = ((self.at[0][:, :, None, None] * self.N[1] + self.at[1][:, None, :, None]) * self.N[2] +
                     self.at[2][:, None, None, :])

    def shift(self, f, a, k, fill):
        """f at + k along axis a: periodic for grains spanning the axis, ``fill`` beyond the window otherwise."""
        r = torch.roll(f, -k, a + 1)
        edge = r.narrow(a + 1, self.w[a] - k if k > 0 else 0, abs(k))
        edge.masked_fill_(~self.full[a][:, None, None, None], fill)
        return r

    def convolve(self, f):
        for a in self.axes:
            if self.w[a] <= RADIUS:
                raise ValueError("a window narrower than the kernel")
            acc = self.taps[RADIUS] * f
            for k in range(1, RADIUS + 1):
                acc += self.taps[RADIUS + k] * (self.shift(f, a, k, -EPS) + self.shift(f, a, -k, -EPS))
            f = acc
        return f

    def top_two(self, p):
        """Largest and second largest function per domain cell and their grains (-inf, G where absent)."""
        cells = self.N[0] * self.N[1] * self.N[2]
        idx = self.cell.reshape(-1)
        ids = torch.arange(self.G, device="cuda")[:, None, None, None].expand(p.shape)
        vals = torch.where(self.inside, p, -math.inf)
        tops = []
        for _ in range(2):
            v = torch.full((cells,), -math.inf, dtype=torch.float64, device="cuda")
            v.scatter_reduce_(0, idx, vals.reshape(-1), "amax")
            hit = (vals == v[self.cell]) & (vals > -math.inf)
            i = torch.full((cells,), self.G, dtype=torch.int64, device="cuda")
            i.scatter_reduce_(0, idx, torch.where(hit, ids, self.G).reshape(-1), "amin")
            tops.append((v, i))
            vals = torch.where(i[self.cell] == ids, -math.inf, vals)
        return tops, ids

    def redistance(self, c):
        pos = c > 0
        a_ = c.abs()
        inv2 = torch.zeros_like(c)
        for a in self.axes:
            big = torch.full_like(c, -1.0)
            for k in (1, -1):
                v = self.shift(c, a, k, -EPS)
                big = torch.where((v > 0) != pos, torch.maximum(big, v.abs()), big)
            inv2 += torch.where(big >= 0, ((a_ + big) / a_) ** 2, 0.0)
        m = torch.where(inv2 > 0, inv2.rsqrt(), EPS)
        m = torch.where(self.inside, m, EPS)
        for _ in range(int(EPS) - 1):
            new = m
            for a in self.axes:
                for k in (1, -1):
                    new = torch.minimum(new, self.shift(m, a, k, EPS) + 1.0)
            m = torch.where(self.inside, new, EPS)
        return torch.where(self.inside & pos, m, -m)

    def box_update(self, f, idf):
        pos = f > 0
        alive = pos.flatten(1).any(1)
        o, n = self.o.clone(), self.n.clone()
        for a in self.axes:
            occ = pos.any([b + 1 for b in range(3) if b != a][1]).any([b + 1 for b in range(3) if b != a][0])
            lo = occ.to(torch.int8).argmax(1)
            hi = self.w[a] - 1 - occ.flip(1).to(torch.int8).argmax(1)
            ext = hi - lo + 1 + 2 * HALO
            was = self.full[a]
            now = ext >= self.N[a]
            o[:, a] = torch.where(now & was, self.o[:, a], (self.o[:, a] + lo - HALO) % self.N[a])
            n[:, a] = torch.where(now, self.N[a], ext)
        o[~alive], n[~alive] = 0, 0
        old_o, old_n, old_w = self.o, self.n, self.w
        self.layout(o, n)
        for a in range(3):
            l = (self.at[a] - old_o[:, a, None]) % self.N[a]
            ok = l < old_n[:, a, None]
            view = [self.G, 1, 1, 1]
            view[a + 1] = -1
            l, ok = torch.where(ok, l, 0).clamp_max(old_w[a] - 1).view(view), ok.view(view)
            size = list(f.shape)
            size[a + 1] = self.w[a]
            f = torch.where(ok, torch.gather(f, a + 1, l.expand(size)), -EPS)
            if idf is not None:
                idf = torch.where(ok, torch.gather(idf, a + 1, l.expand(size)), -1)
        return torch.where(self.inside, f, -EPS), idf

    # starts
    def from_seeds(self, seeds, weights, dims):
        lab = _power_labels(seeds, weights, dims)
        s = torch.as_tensor(np.asarray(seeds)[:, ::-1].copy(), device="cuda")
        w = torch.zeros(self.G, dtype=torch.float64, device="cuda") if weights is None else \
            torch.as_tensor(weights, dtype=torch.float64, device="cuda")
        flat = lab.reshape(-1)
        o = torch.zeros((self.G, 3), dtype=torch.int64, device="cuda")
        n = torch.ones((self.G, 3), dtype=torch.int64, device="cuda")
        for a in self.axes:
            N = self.N[a]
            shape = [1, 1, 1]
            shape[a] = N
            pos = torch.arange(N, device="cuda").view(shape).expand(self.N).reshape(-1)
            r = torch.round(s[:, a]).long() % N
            e = (pos - r[flat]) % N
            e = torch.where(e > N // 2, e - N, e)
            lo = torch.full((self.G,), N, device="cuda").scatter_reduce_(0, flat, e, "amin")
            hi = torch.full((self.G,), -N, device="cuda").scatter_reduce_(0, flat, e, "amax")
            o[:, a] = (r + lo - HALO) % N
            n[:, a] = torch.clamp_max(hi - lo + 1 + 2 * HALO, N)
        gone = torch.bincount(flat, minlength=self.G) == 0
        o[gone], n[gone] = 0, 0
        pairs = []
        for a in self.axes:
            b = torch.roll(lab, -1, a).reshape(-1)
            pairs += [torch.stack([flat, b], 1)[flat != b], torch.stack([b, flat], 1)[flat != b]]
        key = torch.unique(torch.cat(pairs)[:, 0] * self.G + torch.cat(pairs)[:, 1])   # sorted: grain, neighbour
        gi, gj = key // self.G, key % self.G
        cnt = torch.bincount(gi, minlength=self.G)
        rank = torch.arange(len(key), device="cuda") - (torch.cumsum(cnt, 0) - cnt)[gi]
        self.layout(o, n)

        def to_seed(j, a):
            d = self.at[a].double() - s[j, a, None]
            view = [self.G, 1, 1, 1]
            view[a + 1] = -1
            return (d - self.N[a] * torch.round(d / self.N[a])).view(view)

        me = torch.arange(self.G, device="cuda")
        own = [to_seed(me, a) for a in range(3)]
        f = torch.full(self.cell.shape, math.inf, dtype=torch.float64, device="cuda")
        arg = torch.full(self.cell.shape, -1, dtype=torch.int64, device="cuda")
        for k in range(int(cnt.max())):
            j = torch.full((self.G,), -1, dtype=torch.int64, device="cuda")
            j[gi[rank == k]] = gj[rank == k]
            oth = [to_seed(j.clamp_min(0), a) for a in range(3)]
            num = sum(b * b - c * c for b, c in zip(oth, own)) - (w[j.clamp_min(0)] - w)[:, None, None, None]
            den = 2.0 * torch.sqrt(sum((b - c) ** 2 for b, c in zip(oth, own)))
            v = torch.where((j >= 0)[:, None, None, None], num / den, math.inf)
            arg = torch.where(v < f, j[:, None, None, None], arg)
            f = torch.minimum(f, v)
        f = torch.where(self.inside, f.nan_to_num(posinf=EPS).clamp(-EPS, EPS), -EPS)
        return f, torch.where(self.inside, arg, -1)

    def from_labels(self, labels):
        lab = torch.as_tensor(labels, device="cuda").long()
        o = torch.zeros((self.G, 3), dtype=torch.int64)
        n = torch.ones((self.G, 3), dtype=torch.int64)
        gone = (torch.bincount(lab.reshape(-1), minlength=self.G) == 0).cpu()
        for a in self.axes:
            N = self.N[a]
            occ = torch.zeros((self.G, N), dtype=torch.bool, device="cuda")
            shape = [1, 1, 1]
            shape[a] = N
            occ[lab.reshape(-1), torch.arange(N, device="cuda").view(shape).expand(self.N).reshape(-1)] = True
            for g, row in enumerate(occ.cpu().numpy()):      # the longest cyclic run of empty positions
                at = np.flatnonzero(row)
                if len(at) == 0:
                    continue
                gaps = (np.roll(at, -1) - at - 1) % N if len(at) > 1 else np.array([N - 1])
                runs = sorted((-gap, (p + 1) % N) for gap, p in zip(gaps.tolist(), at.tolist()) if gap > 0)
                first, length = (0, N) if not runs else ((runs[0][1] - runs[0][0]) % N, N + runs[0][0])
                o[g, a], n[g, a] = (first - HALO) % N, min(N, length + 2 * HALO)
        o[gone], n[gone] = 0, 0
        self.layout(o.cuda(), n.cuda())
        mine = lab.reshape(-1)[self.cell] == torch.arange(self.G, device="cuda")[:, None, None, None]
        f = torch.where(self.inside & mine, 0.5, -0.5).double()
        return self.redistance(torch.where(self.inside, f, -EPS))


def _pair_weights(quats):
    """(w, M) of every pair: cubic disorientation, Read-Shockley energy, low-angle mobility."""
    q = torch.as_tensor(quats, dtype=torch.float64, device="cuda")
    a, b = q[:, None, :], q[None, :, :]
    aw, ax, ay, az = a[..., 0], -a[..., 1], -a[..., 2], -a[..., 3]
    bw, bx, by, bz = b[..., 0], b[..., 1], b[..., 2], b[..., 3]
    c = torch.stack([aw * bw - ax * bx - ay * by - az * bz, aw * bx + ax * bw + ay * bz - az * by,
                     aw * by - ax * bz + ay * bw + az * bx, aw * bz + ax * by - ay * bx + az * bw], -1).abs()
    c = c.sort(-1, descending=True).values
    best = torch.maximum(c[..., 0], torch.maximum((c[..., 0] + c[..., 1]) / math.sqrt(2.0), 0.5 * c.sum(-1)))
    t = 2.0 * torch.arccos(best.clamp_max(1.0)) / math.radians(THETA_MAX)
    gamma = torch.where(t >= 1.0, 1.0, torch.where(t <= 0.0, 0.0, t * (1.0 - torch.log(t.clamp_min(1e-300)))))
    mob = torch.where(t < 1.0, MOB_LOW, 1.0)
    return (mob * gamma).clamp_min(1e-3), mob


def exact(case, seed):
    if case["kind"] == "serve":
        parts = []
        for k, (n, g, steps) in enumerate(_requests(case)):
            one = _sim("", n, n, n, g, steps, steps)
            parts.append(_exact_sim(one, {"seeds": I.voronoi_seeds(1009 * seed + k, g, (n, n, n))})["volumes"][-1])
        return {"volumes": torch.cat(parts)}
    cells = _box_cells(case["nx"], case["ny"], case["nz"], case["grains"])
    spread = 8.0 if case["start"] == "laguerre" else 3.0       # windows have the largest box's dims
    if cells * spread > 6e8 or cells * spread * case["steps"] > 4.5e10 or \
            (case["physics"] == "read_shockley" and case["grains"] > 4000):
        return None                                            # minutes, or more memory than the card has
    return _exact_sim(case, _arrays(case, seed))


def _exact_sim(case, arrays):
    dims = (case["nx"], case["ny"], case["nz"])
    ms = _Exact(dims, case["grains"])
    physics = case["physics"] != "ideal"
    if case["start"] == "labels":
        f, idf = ms.box_update(ms.from_labels(arrays["labels"]), None)
    else:
        f, idf = ms.from_seeds(arrays["seeds"], arrays.get("weights"), dims)
    if not physics:
        idf = None
    weights = _pair_weights(arrays["quats"]) if case["physics"] == "read_shockley" else None
    energy = torch.as_tensor(arrays["energy"], device="cuda") if case["physics"] == "magnetic" else None
    me = torch.arange(ms.G, device="cuda")[:, None, None, None]
    volumes = []
    for step in range(1, case["steps"] + 1):
        p = ms.convolve(f)
        if physics:
            j = idf.clamp_min(0)
            if weights is not None:
                moved = f + weights[0][me, j] * (p - f)
            else:
                moved = p + (energy[j] - energy[me]) * DT
            p = torch.where(idf >= 0, moved, p)
        p = torch.where(ms.inside, p.clamp(-EPS, EPS), -EPS)
        ((v1, i1), (v2, i2)), ids = ms.top_two(p)
        top = i1[ms.cell] == ids
        m = torch.where(top, v2[ms.cell], v1[ms.cell]).clamp_min(-EPS)
        if physics:
            idf = torch.where(top, i2[ms.cell], i1[ms.cell])
            idf = torch.where(ms.inside & (m > -EPS), idf, -1)
        f = ms.redistance(torch.where(ms.inside, 0.5 * (p - m), -EPS))
        if step % case["every"] == 0 or step == case["steps"]:
            volumes.append((f + 0.5).clamp(0.0, 1.0).flatten(1).sum(1))
        f, idf = ms.box_update(f, idf)
    out = {"volumes": torch.stack(volumes), "owner": None}
    if case["state"]:
        out["boxes"] = None
        phi = f[ms.inside]
        out["phi"] = torch.zeros(_phi_room(case), dtype=torch.float64, device="cuda")
        out["phi"][:phi.numel()] = phi
    return out
