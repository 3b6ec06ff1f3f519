"""Performance cases of the particle-in-cell library, called as a user's program calls it.

Families (key "kind"):
  step     steps of one run, 2D or 3D, then its diagnostics history and fields (and, for the
           closure study, the coarse moments every few steps).  "fresh": a pass is a whole short
           run from host arrays (engine, load, steps, read-back), as small runs are made; else
           one stretch of a long run on an engine that is kept
  scan     steps of a batch of independent 2D runs of different grids and temperatures
  record   one coarse-moment snapshot of a 3D state
  hybrid   steps of the quasi-neutral hybrid model, then its energies, a and beta_p
  forward  the closure network on a batch of samples
  train    one full-batch training step of the closure network

`exact` is a plain float64 restatement of each path in torch (collisions excepted).
"""
import ctypes
import math

import numpy as np
import torch

import paper_0808_4078_gb300 as pic

DX, DT, GAMMA_B, NB = 0.1, 0.05, 3.0, 0.1
EXACT_LIMIT = 1.2e9      # particle steps (times the terms of a 3D move) that `exact` takes on


# ------------------------------------------------------------------ cases
def _step(name, nx, ny, ppc, steps, nz=1, T=0.1, Tbg=0.001, nu=0.0, coll=0.0, filt=0, diag=1, record=0, fresh=0,
          ids=0):
    return dict(name=name, kind="step", nx=nx, ny=ny, nz=nz, ppc=ppc, steps=steps, T=T, Tbg=Tbg, nu=nu, coll=coll,
                filt=filt, diag=diag, record=record, fresh=fresh, ids=ids)


def listed():
    return [
        # a cold beam on a small grid, the size of a first run or a test, with its particles read
        # back by id: launches and latency
        _step("run2d_64x64_cold", 64, 64, 16, 500, T=0.0, Tbg=0.0, fresh=1, ids=1),
        # the crop on which the growth rate of the warm Krook run is followed, every step recorded
        _step("run2d_128x128_krook", 128, 128, 64, 240, nu=0.1, fresh=1),
        # an odd grid with the options on: binary collisions of the return current, current filter
        _step("run2d_336x208_collide_filter", 336, 208, 27, 120, coll=0.15, filt=1, fresh=1),
        # the headline run: warm beam, Krook drag on the return current, 134M particles
        _step("step2d_1024x1024_krook", 1024, 1024, 64, 24, nu=0.1, diag=10),
        # 3D with Krook drag on the return current, ragged grid and particle count
        _step("run3d_40x48x36_krook", 40, 48, 11, 120, nz=36, nu=0.15, diag=4, fresh=1),
        # the 3D crop of the closure study: current filter, moments recorded every 4 steps
        _step("step3d_64x64x128_closure", 64, 64, 8, 16, nz=128, T=0.2, Tbg=0.0, filt=1, record=4),
        # the 3D hot beam, 67M particles
        _step("step3d_128x128x256_hot", 128, 128, 8, 24, nz=256, T=0.2, Tbg=0.0, diag=10),
        # the temperature and collision-rate scan: runs of mixed grids stepped as one batch
        dict(name="scan2d_24runs", kind="scan", runs=24, div=2, ppc=32, steps=16, diag=10),
        # one snapshot of the moment recorder on a 3D state
        dict(name="record3d_128x128x256", kind="record", nx=128, ny=128, nz=256, ppc=8, bx=4, by=4),
        # the hybrid model at its benchmark size
        dict(name="hybrid_1024x1024", kind="hybrid", nx=1024, ny=1024, ppc=16, steps=96, nu=0.1),
        # inference on the coarse cells of many snapshots
        dict(name="forward_1048576", kind="forward", n=1 << 20, nin=9),
        # one Adam step on the full-size closure training set (a ragged sample count)
        dict(name="train_403938", kind="train", n=403938, nin=9),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _multiple(rng, lo, hi, m):
    return m * max(1, round(_log(rng, lo, hi) / m))


def draw(rng):
    kind = rng.choice(["step2d", "step2d", "step3d", "step3d", "scan", "record", "hybrid", "forward", "train"])
    if kind == "step2d":
        nx, ny, ppc = _multiple(rng, 16, 1024, 16), _multiple(rng, 16, 1024, 16), round(_log(rng, 2, 64))
        opt = rng.choice(["plain", "krook", "collide"])
        c = _step("", nx, ny, ppc, rng.choice([8, 16, 21]), T=rng.uniform(0.0, 1.0), nu=0.1 if opt == "krook" else 0.0,
                  coll=0.15 if opt == "collide" else 0.0, filt=rng.choice([0, 1]), diag=rng.choice([1, 10]))
        if nx * ny * ppc < 4 << 20:
            c.update(fresh=1, steps=rng.choice([100, 131, 240]))
    elif kind == "step3d":
        nx, ny, nz = _multiple(rng, 16, 128, 8), _multiple(rng, 16, 128, 8), _multiple(rng, 16, 256, 4)
        opt = rng.choice(["plain", "plain", "krook", "collide"])
        c = _step("", nx, ny, round(_log(rng, 2, 8)), rng.choice([8, 13, 16]), nz=nz, T=rng.uniform(0.05, 0.4),
                  nu=0.15 if opt == "krook" else 0.0, coll=0.15 if opt == "collide" else 0.0,
                  filt=rng.choice([0, 1]), diag=rng.choice([1, 10]), record=rng.choice([0, 4]))
        if nx * ny * nz * c["ppc"] < 3 << 20:
            c.update(fresh=1, steps=rng.choice([64, 93, 120]))
    elif kind == "scan":
        c = dict(kind="scan", runs=rng.randint(3, 24), div=rng.choice([2, 4, 8]), ppc=round(_log(rng, 4, 32)),
                 steps=rng.choice([8, 13, 16]), diag=rng.choice([1, 10]))
    elif kind == "record":
        c = dict(kind="record", nx=_multiple(rng, 16, 128, 16), ny=_multiple(rng, 16, 128, 16),
                 nz=_multiple(rng, 16, 256, 4), ppc=round(_log(rng, 2, 8)), bx=rng.choice([2, 4, 8]),
                 by=rng.choice([2, 4, 8]))
    elif kind == "hybrid":
        c = dict(kind="hybrid", nx=1 << rng.randint(4, 10), ny=1 << rng.randint(4, 10), ppc=round(_log(rng, 2, 16)),
                 steps=rng.choice([16, 37, 64]), nu=rng.choice([0.0, 0.1]))
    else:
        c = dict(kind=kind, n=round(_log(rng, 200, 1 << 20 if kind == "forward" else 403938)), nin=rng.choice([8, 9]))
    c.pop("name", None)
    return c


def work(case):
    """Per step a particle's offsets, momenta (and in 3D its cell) are read and written, the
    fields read and written and the current written and read once."""
    k = case["kind"]
    if k in ("step", "scan", "record"):
        if k == "scan":
            cells, nd, ppc = sum(nx * ny for nx, ny, _, _ in _scan_table(case)), 2, case["ppc"]
        else:
            cells, nd, ppc = case["nx"] * case["ny"] * case["nz"], 2 if case["nz"] == 1 else 3, case["ppc"]
        n = 2 * cells * ppc
        if k == "record":
            return dict(bytes=28.0 * n + 24.0 * cells, flops=60.0 * n)
        per = 40.0 if nd == 2 else 56.0
        return dict(bytes=float(case["steps"] * (per * n + 96.0 * cells)),
                    flops=float(case["steps"] * ((230 if nd == 2 else 420) * n + 60 * cells)))
    if k == "hybrid":
        cells = case["nx"] * case["ny"]
        n = cells * case["ppc"]
        return dict(bytes=float(case["steps"] * (44.0 * n + 150.0 * cells)),
                    flops=float(case["steps"] * (110 * n + 400 * cells)))
    n = case["n"]
    mac = 9 * 64 + 64 * 64 + 64
    if k == "forward":
        return dict(bytes=40.0 * n, flops=2.0 * mac * n)
    return dict(bytes=40.0 * n, flops=6.0 * mac * n)


# ------------------------------------------------------------------ inputs
def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _species(g, nd, ncell, ppc, T, Tbg):
    """Beam and background of a Weibel load on the GPU: [(w, cell, offset, u)] with the
    background drift chosen so that the sampled current along z vanishes."""
    out = []
    uz0 = math.sqrt(GAMMA_B * GAMMA_B - 1.0)
    current = 0.0
    for s, (density, temp) in enumerate(((NB, T), (1.0 - NB, Tbg))):
        n, w = ncell * ppc, density / ppc
        cell = torch.arange(ncell, dtype=torch.int32, device="cuda").repeat_interleave(ppc)
        off = torch.rand((nd, n), generator=g, device="cuda")
        u = torch.randn((3, n), generator=g, device="cuda") * math.sqrt(temp) if temp > 0 else \
            torch.zeros((3, n), device="cuda")
        if s == 0:
            u[2] = uz0
            current = w * float((u[2] / (1 + (u * u).sum(0)).sqrt()).double().sum())
        else:
            d = 0.0
            for _ in range(8):
                uz = u[2] + d
                t = 1 + u[0] ** 2 + u[1] ** 2
                gam = (t + uz * uz).sqrt()
                d -= (float((uz / gam).double().sum()) + current / w) / float((t / gam ** 3).double().sum())
            u[2] += d
        out.append((w, cell, off, u))
    return out


def _host(t):
    return t.cpu().numpy()


def _scan_table(case):
    """Grids, temperature and Krook rate of the scan's runs: sides from 128..512 over `div`."""
    rng = np.random.default_rng(4)
    sides = [s // case["div"] for s in (128, 192, 256, 384, 512)]
    sides = [max(16, s // 16 * 16) for s in sides]
    return [(int(rng.choice(sides)), int(rng.choice(sides)), float(rng.random()),
             float(rng.choice((0.0, 0.01, 0.1, 1.0)))) for _ in range(case["runs"])]


def _records(case):
    return max(1, -(-case["steps"] // case["diag"]))


def _arrays(case, seed):
    """Host arrays of both species: (w, nu, cell, offset, u)."""
    nd = 2 if case["nz"] == 1 else 3
    sp = _species(_generator(seed), nd, case["nx"] * case["ny"] * case["nz"], case["ppc"], case.get("T", 0.2),
                  case.get("Tbg", 0.0))
    return [(w, case.get("nu", 0.0) if s == 1 else 0.0, _host(cell), _host(off), _host(u))
            for s, (w, cell, off, u) in enumerate(sp)]


def _engine(case, arrays):
    coll = case.get("coll", 0.0)
    eng = pic.Engine(2 if case["nz"] == 1 else 3, case["nx"], case["ny"], case["nz"], dx=DX, dt=DT,
                     capacity=[a[2].shape[0] for a in arrays], diag_interval=case.get("diag", 1),
                     diag_capacity=_records(case) if "steps" in case else 8,
                     track_ids=coll > 0 or case.get("ids", 0), j_filter=case.get("filt", 0))
    for s, (w, nu, cell, off, u) in enumerate(arrays):
        eng.load_species(s, -1.0, 1.0, w, nu, cell, off, u)
        if coll > 0 and s == 1:          # the return current's electrons collide with the ions
            eng.set_collisions(s, coll, 77)
    return eng


def _hybrid_load(case, seed):
    g = _generator(seed)
    nx, ny, ppc = case["nx"], case["ny"], case["ppc"]
    n = nx * ny * ppc
    cell = torch.arange(nx * ny, device="cuda").repeat_interleave(ppc)
    off = torch.rand((2, n), generator=g, device="cuda").double()
    u = (torch.randn((2, n), generator=g, device="cuda") * math.sqrt(0.1)).double()
    uz = torch.full((n,), float(np.float32(math.sqrt(GAMMA_B ** 2 - 1))), dtype=torch.float64, device="cuda")
    bz = uz / (1 + u[0] ** 2 + u[1] ** 2 + uz * uz).sqrt()
    return (cell % nx) + off[0], (cell // nx) + off[1], u[0], u[1], uz, -NB * float(bz.mean()) / (1 - NB)


# means and spreads of the recorder's rows 0..8 in a hot-beam state
_MU = np.array([0.1, 0.9, 2.8, -0.1, 0.2, 0.02, 0.001, 0.001, 0.0005])
_SD = np.array([0.02, 0.02, 0.1, 0.03, 0.05, 0.02, 0.0005, 0.0005, 0.0003])


def _network(seed, nin):
    g = np.random.default_rng(seed)
    w1 = g.uniform(-1, 1, (64, 9)) / math.sqrt(nin)
    w1[:, nin:] = 0.0
    parts = [w1.ravel(), g.uniform(-1, 1, 64) / math.sqrt(nin), g.uniform(-1, 1, 64 * 64) / 8.0,
             g.uniform(-1, 1, 64) / 8.0, g.uniform(-1, 1, 64) / 8.0, [0.0]]
    return np.concatenate(parts).astype(np.float32)


def _samples(case, seed):
    g = _generator(seed)
    z = torch.randn((9, case["n"]), generator=g, device="cuda")
    sd, mu = (torch.tensor(v, dtype=torch.float32, device="cuda")[:, None] for v in (_SD, _MU))
    t = 0.05 * torch.tanh(z[0] - 0.5 * z[3] + z[8]) + 0.02 * torch.randn(case["n"], generator=g, device="cuda")
    return z * sd + mu, t


def prepare(case, seed):
    k = case["kind"]
    if k == "step":
        arrays = _arrays(case, seed)
        return dict(case=case, arrays=arrays) if case["fresh"] else dict(case=case, eng=_engine(case, arrays))
    if k == "scan":
        table = _scan_table(case)
        caps = [nx * ny * case["ppc"] for nx, ny, _, _ in table]
        eng = pic.Engine(2, dx=DX, dt=DT, runs=[(nx, ny, 1, (c, c)) for (nx, ny, _, _), c in zip(table, caps)],
                         diag_interval=case["diag"], diag_capacity=_records(case))
        g = _generator(seed)
        for r, (nx, ny, T, nu) in enumerate(table):
            for s, (w, cell, off, u) in enumerate(_species(g, 2, nx * ny, case["ppc"], T, 0.001)):
                eng.load_species(s, -1.0, 1.0, w, nu if s == 1 else 0.0, _host(cell), _host(off), _host(u), run=r)
        return dict(case=case, eng=eng)
    if k == "record":
        eng = _engine(case, _arrays(case, seed))
        eng.step(4)
        eng.sync()
        return dict(case=case, eng=eng)
    if k == "hybrid":
        n = case["nx"] * case["ny"] * case["ppc"]
        eng = pic.HybridEngine(case["nx"], case["ny"], DX, DX, DT, 1.0, case["nu"], NB / case["ppc"], n)
        X, Y, ux, uy, uz, bp = _hybrid_load(case, seed)
        eng.load(*(_host(v) for v in (X, Y, ux, uy, uz)), bp)
        return dict(case=case, eng=eng)
    x, t = _samples(case, seed)
    net = pic.ClosureNet(_network(seed, case["nin"]), _MU, _SD, nin=case["nin"])
    torch.cuda.synchronize()
    return dict(case=case, net=net, x=x, t=t)


# ------------------------------------------------------------------ one pass
def _history(recs):
    return {k: np.array([r[k] for r in recs]) for k in ("WE", "WB", "Ekin", "P")}


def _moments(rows):
    return {name: rows[:, i] for i, name in enumerate(pic.MOMENT_ROWS)}


def run(state):
    case = state["case"]
    k = case["kind"]
    if k == "step":
        eng, out = _engine(case, state["arrays"]) if case["fresh"] else state["eng"], {}
        every = case["record"]
        if every:
            rows = []
            for _ in range(case["steps"] // every):
                eng.step(every)
                rows.append(eng.record_moments(4, 4))
            eng.step(case["steps"] % every)
            out.update(_moments(torch.stack(rows)))
        else:
            eng.step(case["steps"])
        out.update(_history(eng.diag()))
        out["E"], out["B"], _ = eng.fields()
        if case["ids"]:
            for s in range(2):
                cell, off, u, ids = eng.particles(s)
                at = np.argsort(ids)
                out[f"cell{s}"], out[f"offset{s}"], out[f"u{s}"] = cell[at], off[:, at], u[:, at]
        if case["fresh"]:
            eng.close()
        return out
    if k == "scan":
        eng = state["eng"]
        eng.step(case["steps"])
        hist = [_history(eng.diag(run=r)) for r in range(len(eng.runs))]
        out = {key: np.stack([h[key] for h in hist]) for key in hist[0]}
        for r in (0, len(eng.runs) - 1):
            out[f"E{r}"], out[f"B{r}"], _ = eng.fields(run=r)
        return out
    if k == "record":
        return _moments(state["eng"].record_moments(case["bx"], case["by"])[None])
    if k == "hybrid":
        eng = state["eng"]
        eng.step(case["steps"])
        a, bp = (np.empty((case["ny"], case["nx"])) for _ in range(2))
        vp = ctypes.c_void_p
        rc = pic.lib().pic_hybrid_get(eng._h, a.ctypes.data_as(vp), bp.ctypes.data_as(vp), None, None, None, None)
        assert rc == 0
        return dict(a=a, beta_p=bp, energies=eng.energies())
    net = state["net"]
    if k == "forward":
        return net.forward(state["x"])
    loss = net.train_step(state["x"], state["t"], 1e-3)
    return dict(loss=loss, params=net.params, m=net.m, v=net.v)


# ------------------------------------------------------------------ float64 restatement
class _Plasma:
    """The explicit step in float64: CIC gather, Boris, drag, move, Esirkepov deposit, Yee.
    Arrays [nz][ny][nx]; axis 0, 1, 2 = x, y, z; a species is (w, nu, cell per axis, offset, u)."""

    def __init__(self, shape, species, nd, filt):
        self.n = shape                       # (nx, ny, nz)
        self.nd, self.filt = nd, filt
        dims = (shape[2], shape[1], shape[0])
        self.E, self.B = ([torch.zeros(dims, dtype=torch.float64, device="cuda") for _ in range(3)] for _ in range(2))
        self.sp = []
        for w, nu, cell, off, u in species:
            c = cell.long()
            ax = [c % shape[0], c // shape[0] % shape[1], c // (shape[0] * shape[1])][:nd]
            self.sp.append(dict(w=w, nu=nu, c=ax, o=[o.double() for o in off], u=[v.double() for v in u], ub=None))
        for s in self.sp:
            self._means(s)

    def _index(self, ijk):
        f = ijk[0] % self.n[0] + self.n[0] * (ijk[1] % self.n[1])
        return f + self.n[0] * self.n[1] * (ijk[2] % self.n[2]) if self.nd == 3 else f

    def _means(self, s):
        if s["nu"] <= 0:
            return
        nc = self.n[0] * self.n[1] * self.n[2]
        g = self._index(s["c"])
        cnt = torch.bincount(g, minlength=nc).clamp(min=1)
        s["ub"] = [torch.zeros(nc, dtype=torch.float64, device="cuda").index_add_(0, g, v) / cnt for v in s["u"]]

    def _interp(self, F, half, c, o):
        base, wt = [], []
        for a in range(self.nd):
            d = o[a] - 0.5 if half[a] else o[a]
            fl = torch.floor(d)
            base.append(c[a] + fl.long())
            wt.append((1 - (d - fl), d - fl))
        F = F.reshape(-1)
        out = 0.0
        for corner in range(1 << self.nd):
            bit = [corner >> a & 1 for a in range(self.nd)]
            w = wt[0][bit[0]]
            for a in range(1, self.nd):
                w = w * wt[a][bit[a]]
            out = out + w * F[self._index([base[a] + bit[a] for a in range(self.nd)])]
        return out

    def fields_at(self, c, o):
        e = [self._interp(self.E[q], [a == q for a in range(3)], c, o) for q in range(3)]
        b = [self._interp(self.B[q], [a != q for a in range(3)], c, o) for q in range(3)]
        return e, b

    def _push(self, s, sl, J, rec, index):
        c, o, u0 = ([v[sl] for v in s[k]] for k in ("c", "o", "u"))
        e, b = self.fields_at(c, o)
        h = -0.5 * DT
        um = [u0[a] + h * e[a] for a in range(3)]
        g = torch.sqrt(1 + um[0] ** 2 + um[1] ** 2 + um[2] ** 2)
        t = [h * v / g for v in b]
        f = 2 / (1 + t[0] ** 2 + t[1] ** 2 + t[2] ** 2)
        up = [um[a] + um[(a + 1) % 3] * t[(a + 2) % 3] - um[(a + 2) % 3] * t[(a + 1) % 3] for a in range(3)]
        u = [um[a] + f * (up[(a + 1) % 3] * t[(a + 2) % 3] - up[(a + 2) % 3] * t[(a + 1) % 3]) + h * e[a]
             for a in range(3)]
        if s["ub"] is not None:
            cell = self._index(c)
            u = [u[a] + math.expm1(-s["nu"] * DT) * s["ub"][a][cell] for a in range(3)]
        gam = torch.sqrt(1 + u[0] ** 2 + u[1] ** 2 + u[2] ** 2)
        if rec is not None:
            m = [0.5 * (u0[a] + u[a]) for a in range(3)]
            k = torch.sqrt(1 + m[0] ** 2 + m[1] ** 2 + m[2] ** 2) - 1
            rec["Ekin"][index] += s["w"] * float(k.sum())
            for a in range(3):
                rec["P"][a] += s["w"] * float(m[a].sum())
        S0, S1, C, base = [], [], [], []
        for a in range(self.nd):
            r = o[a] + u[a] / gam * (DT / DX)
            st = torch.floor(r)
            low = torch.clamp(st, max=0.0)
            S0.append([torch.clamp(1 - (o[a] - low - k).abs(), min=0) for k in range(3)])
            S1.append([torch.clamp(1 - (r - low - k).abs(), min=0) for k in range(3)])
            d0 = S1[a][0] - S0[a][0]
            C.append([d0, d0 + S1[a][1] - S0[a][1]])
            base.append(c[a] + low.long())
            s["o"][a][sl] = r - st
            s["c"][a][sl] = (c[a] + st.long()) % self.n[a]
        for a in range(3):
            s["u"][a][sl] = u[a]
        flux = s["w"] * DX / DT              # -q w dx / dt for q = -1

        def add(q, ijk, v):
            J[q].index_add_(0, self._index([base[a] + ijk[a] for a in range(self.nd)]), v)

        def shape2(p, q, i, j):              # path average of S_p(i) S_q(j)
            return S0[p][i] * (S0[q][j] / 3 + S1[q][j] / 6) + S1[p][i] * (S0[q][j] / 6 + S1[q][j] / 3)

        if self.nd == 3:
            for q in range(3):
                p1, p2 = (q + 1) % 3, (q + 2) % 3
                for i in range(3):
                    for j in range(3):
                        f = flux * shape2(p1, p2, i, j)
                        for k in range(2):
                            ijk = [0, 0, 0]
                            ijk[q], ijk[p1], ijk[p2] = k, i, j
                            add(q, ijk, f * C[q][k])
            return
        for j in range(3):
            for k in range(2):
                add(0, (k, j), flux * C[0][k] * 0.5 * (S0[1][j] + S1[1][j]))
                add(1, (j, k), flux * C[1][k] * 0.5 * (S0[0][j] + S1[0][j]))
            for i in range(3):
                add(2, (i, j), -s["w"] * (u[2] / gam) * shape2(0, 1, i, j))

    def _curl(self, F, sign):
        """sign +1: forward differences (curl E), -1: backward differences (curl B), times dx."""
        def d(f, axis):
            if axis == 2 and self.nd == 2:
                return torch.zeros_like(f)
            return sign * (torch.roll(f, -sign, 2 - axis) - f)
        return [d(F[(a + 2) % 3], (a + 1) % 3) - d(F[(a + 1) % 3], (a + 2) % 3) for a in range(3)]

    def step(self, record):
        dV = DX ** self.nd
        rec = None
        if record:
            rec = dict(WE=[float((f * f).sum()) * dV for f in self.E], WB=[float((f * f).sum()) * dV for f in self.B],
                       Ekin=[0.0] * len(self.sp), P=[0.0] * 3)
        J = [torch.zeros(self.E[0].numel(), dtype=torch.float64, device="cuda") for _ in range(3)]
        for i, s in enumerate(self.sp):
            n = s["o"][0].numel()
            for a in range(0, n, 1 << 22):
                self._push(s, slice(a, min(n, a + (1 << 22))), J, rec, i)
            self._means(s)
        J = [j.reshape(self.E[0].shape) for j in J]
        if self.filt:
            for axis in range(self.nd):
                J = [0.25 * (torch.roll(j, 1, 2 - axis) + 2 * j + torch.roll(j, -1, 2 - axis)) for j in J]
        r = DT / DX
        for phase in range(3):
            if phase == 1:
                cb = self._curl(self.B, -1)
                self.E = [self.E[a] + r * cb[a] - DT * J[a] for a in range(3)]
            else:
                ce = self._curl(self.E, 1)
                self.B = [self.B[a] - 0.5 * r * ce[a] for a in range(3)]
        if rec is not None:
            rec["Ekin"] = [v * dV for v in rec["Ekin"]]
            rec["P"] = [v * dV for v in rec["P"]]
        return rec

    def moments(self, bx, by):
        ncx, ncy = self.n[0] // bx, self.n[1] // by
        nc = ncx * ncy
        out = torch.zeros((12, nc), dtype=torch.float64, device="cuda")

        def total(i, v):
            return torch.zeros(nc, dtype=torch.float64, device="cuda").index_add_(0, i, v)

        def block(F):
            return F.mean(0).reshape(ncy, by, ncx, bx).mean((1, 3)).reshape(-1)

        for k, s in enumerate(self.sp):
            i = s["c"][1] // by * ncx + s["c"][0] // bx
            cnt = torch.bincount(i, minlength=nc).double()
            mean = [total(i, v) / cnt for v in s["u"]]
            var = [total(i, (v - m[i]) ** 2) / cnt for v, m in zip(s["u"], mean)]
            out[k] = s["w"] * cnt / (bx * by * self.n[2])
            out[2 + k] = mean[2]
            out[4 + 2 * k] = 0.5 * (var[0] + var[1])
            out[5 + 2 * k] = var[2]
        if self.nd == 3:
            out[8] = block(sum((f - f.mean(0, keepdim=True)) ** 2 for f in self.E))
        F, V = torch.zeros_like(cnt), [torch.zeros_like(cnt) for _ in range(2)]
        n = i.numel()
        for a in range(0, n, 1 << 22):
            sl = slice(a, min(n, a + (1 << 22)))
            c, o, u = ([v[sl] for v in s[k]] for k in ("c", "o", "u"))
            e, b = self.fields_at(c, o)
            g = torch.sqrt(1 + u[0] ** 2 + u[1] ** 2 + u[2] ** 2)
            F += total(i[sl], -(e[2] + u[0] / g * b[1] - u[1] / g * b[0]))
            for a2 in range(2):
                V[a2] += total(i[sl], u[a2] / g)
        out[9] = F / cnt
        out[10] = -(block(self.E[2]) + V[0] / cnt * block(self.B[1]) - V[1] / cnt * block(self.B[0]))
        out[11] = s["nu"] + (out[10] - out[9]) / out[3]
        return out


def _plasma(nx, ny, nz, species, nu, filt=0):
    return _Plasma((nx, ny, nz), [(w, nu if i == 1 else 0.0, c, o, u) for i, (w, c, o, u) in enumerate(species)],
                   2 if nz == 1 else 3, filt)


def _np(fs):
    return np.stack([f.reshape(-1).cpu().numpy() for f in fs])


def _exact_moments(rows):
    out = _moments(rows)
    out["nu_eff"] = None                         # a ratio of small differences: its parts are compared
    return out


def _exact_step(case, seed):
    p = _plasma(case["nx"], case["ny"], case["nz"],
                _species(_generator(seed), 2 if case["nz"] == 1 else 3, case["nx"] * case["ny"] * case["nz"],
                         case["ppc"], case["T"], case["Tbg"]), case["nu"], case["filt"])
    recs, rows = [], []
    for n in range(case["steps"]):
        r = p.step(n % case["diag"] == 0)
        if r:
            recs.append(r)
        if case["record"] and (n + 1) % case["record"] == 0:
            rows.append(p.moments(4, 4))
    out = _exact_moments(torch.stack(rows)) if case["record"] else {}
    out.update(_history(recs))
    out["E"], out["B"] = _np(p.E), _np(p.B)
    if case["ids"]:
        for i, s in enumerate(p.sp):
            # a particle within rounding of a cell edge may count to either side
            out[f"cell{i}"], out[f"offset{i}"], out[f"u{i}"] = None, None, _np(s["u"])
    return out


def _exact_scan(case, seed):
    g, hist, out = _generator(seed), [], {}
    table = _scan_table(case)
    for r, (nx, ny, T, nu) in enumerate(table):
        p = _plasma(nx, ny, 1, _species(g, 2, nx * ny, case["ppc"], T, 0.001), nu)
        recs = [p.step(n % case["diag"] == 0) for n in range(case["steps"])]
        hist.append(_history([v for v in recs if v]))
        if r in (0, len(table) - 1):
            out[f"E{r}"], out[f"B{r}"] = _np(p.E), _np(p.B)
    out.update({key: np.stack([h[key] for h in hist]) for key in hist[0]})
    return out


def _exact_hybrid(case, seed):
    nx, ny, nu, w = case["nx"], case["ny"], case["nu"], NB / case["ppc"]
    X, Y, ux, uy, P, bp0 = _hybrid_load(case, seed)
    i, j = X.floor().long(), Y.floor().long()
    fx, fy = X - i, Y - j
    del X, Y
    a = torch.zeros((ny, nx), dtype=torch.float64, device="cuda")
    bp = torch.full_like(a, bp0)
    kx, ky = (torch.sin(math.pi * torch.arange(n, device="cuda", dtype=torch.float64) / n) ** 2 for n in (nx, ny))
    lam = -(4 / DX ** 2) * (ky[:, None] + kx[None, :])
    nbar = 1.0 - NB

    def corners():
        i1, j1 = (i + 1) % nx, (j + 1) % ny
        return ((j * nx + i, (1 - fx) * (1 - fy)), (j * nx + i1, fx * (1 - fy)), (j1 * nx + i, (1 - fx) * fy),
                (j1 * nx + i1, fx * fy))

    def interp(F):
        F = F.reshape(-1)
        return sum(wt * F[c] for c, wt in corners())

    def deposit(q):
        out = torch.zeros(nx * ny, dtype=torch.float64, device="cuda")
        for c, wt in corners():
            out.index_add_(0, c, q * wt)
        return out.reshape(ny, nx)

    def lap(F):
        return (sum(torch.roll(F, s, d) for s in (1, -1) for d in (0, 1)) - 4 * F) / DX ** 2

    def energy():
        uz = P + interp(a)
        g = torch.sqrt(1 + ux ** 2 + uy ** 2 + uz ** 2)
        return [0.5 * float(sum((torch.roll(a, -1, d) - a) ** 2 for d in (0, 1)).sum()),
                w * float((g - 1).sum()) * DX * DX, 0.5 * float((npl * bp ** 2).sum()) * DX * DX]

    npl = None
    for _ in range(case["steps"]):
        f = a.reshape(-1)
        (c0, _), (c1, _), (c2, _), (c3, _) = corners()
        gx = ((1 - fy) * (f[c1] - f[c0]) + fy * (f[c3] - f[c2])) / DX
        gy = ((1 - fx) * (f[c2] - f[c0]) + fx * (f[c3] - f[c1])) / DX
        uz = P + interp(a)
        q = uz / torch.sqrt(1 + ux ** 2 + uy ** 2 + uz ** 2) - interp(bp)
        ux, uy = ux - DT * q * gx, uy - DT * q * gy
        g = torch.sqrt(1 + ux ** 2 + uy ** 2 + uz ** 2)
        fx, fy = fx + DT / DX * ux / g, fy + DT / DX * uy / g
        si, sj = fx.floor(), fy.floor()
        i, j, fx, fy = (i + si.long()) % nx, (j + sj.long()) % ny, fx - si, fy - sj
        uz = P + interp(a)
        jb = deposit(w * uz / torch.sqrt(1 + ux ** 2 + uy ** 2 + uz ** 2))
        npl = (1.0 - deposit(torch.full_like(fx, w))).clamp(min=0)
        r = jb + npl * (bp - nu * DT * bp) - lap(a)
        d, p, rz, r0 = torch.zeros_like(a), None, None, float((r * r).sum())
        for _ in range(60):
            z = torch.fft.ifft2(torch.fft.fft2(r) / (lam - nbar)).real
            new = float((r * z).sum())
            p = z if p is None else z + new / rz * p
            rz = new
            ap = lap(p) - npl * p
            al = rz / float((p * ap).sum())
            d, r = d + al * p, r - al * ap
            if float((r * r).sum()) <= 1e-26 * r0:
                break
        bp = bp + d - nu * DT * bp
        a = a + d
    return dict(a=a.cpu().numpy(), beta_p=bp.cpu().numpy(), energies=np.array(energy()))


def _exact_net(case, seed):
    x, t = _samples(case, seed)
    par = torch.tensor(_network(seed, case["nin"]), device="cuda").double()
    sizes = (("W1", (64, 9)), ("b1", (64,)), ("W2", (64, 64)), ("b2", (64,)), ("w3", (64,)), ("b3", (1,)))
    P, at = {}, 0
    for name, shape in sizes:
        P[name] = par[at:at + math.prod(shape)].reshape(shape)
        at += math.prod(shape)

    def bf(v):
        return v.float().bfloat16().double()

    def dsilu(z):
        s = torch.sigmoid(z)
        return s * (1 + z * (1 - s))

    mu, sd = (torch.tensor(v.astype(np.float32), device="cuda").double()[:, None] for v in (_MU, _SD))
    xn = ((x.double() - mu) / sd).T
    xn[:, case["nin"]:] = 0.0
    xn = bf(xn)
    z1 = xn @ bf(P["W1"]).T + P["b1"]
    h1 = bf(z1 * torch.sigmoid(z1))
    z2 = h1 @ bf(P["W2"]).T + P["b2"]
    h2 = z2 * torch.sigmoid(z2)
    y = h2 @ P["w3"] + P["b3"]
    if case["kind"] == "forward":
        return y
    res = y - t.double()
    dy = 2 * res / case["n"]
    d2 = dy[:, None] * P["w3"] * dsilu(z2)
    d1 = bf(d2) @ bf(P["W2"]) * dsilu(z1)
    g = torch.cat([(d1.T @ xn).reshape(-1), d1.sum(0), (d2.T @ h1).reshape(-1), d2.sum(0), h2.T @ dy, dy.sum()[None]])
    m, v = 0.1 * g, 0.001 * g * g
    return dict(loss=float((res * res).mean()), params=par - 1e-3 * (m / 0.1) / (torch.sqrt(v / 0.001) + 1e-8), m=m, v=v)


def exact(case, seed):
    k = case["kind"]
    if k in ("forward", "train"):
        return _exact_net(case, seed)
    if case.get("coll", 0.0) > 0:
        return None                              # keyed random draws
    if k == "hybrid":
        return _exact_hybrid(case, seed)
    if work(case)["flops"] / 230 > EXACT_LIMIT:
        return None
    if k == "scan":
        return _exact_scan(case, seed)
    if k == "step":
        return _exact_step(case, seed)
    p = _plasma(case["nx"], case["ny"], case["nz"],
                _species(_generator(seed), 3, case["nx"] * case["ny"] * case["nz"], case["ppc"], 0.2, 0.0), 0.0)
    for _ in range(4):
        p.step(False)
    return _exact_moments(p.moments(case["bx"], case["by"])[None])
