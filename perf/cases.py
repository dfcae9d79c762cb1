"""The work that programs have this library do, as measurable cases.

A case is one call (or the few calls that belong together) through the public entry
points, on catalogues of a survey's or a simulation's shape.  ``prepare`` makes what a
program has in hand before the call: the catalogue on the device (on the host for the
host-buffer entry point) and the plan, batch or network that it keeps.  ``run`` is one
pass.  ``exact`` is the same quantity in 64 bits from plain torch.

The multipoles are returned in float32: the meshes and transforms behind them are
float32, and a data vector is kept in that type.  k, the mode counts, alpha, I and S/I
are float64, as in the result row.
"""
import math

import numpy as np
import torch

import paper_1505_05341_gb300 as ys

BOXES = {  # box_min, box_len; the observer sits at the origin
    "cube": ((350.0, 350.0, 350.0), 500.0),         # a simulation cube away from the observer
    "cone": ((-20.0, -20.0, -20.0), 2000.0),        # a 60 degree cone about (1, 1, 1), r in [300, 2100)
    "shell": ((-1750.0, -1750.0, -1750.0), 3500.0),  # full sky, r in [600, 2000) clipped to the box
    "cap": ((-1750.0, -1750.0, -437.0), 3500.0),    # 7000 deg^2 about +z, r in [1100, 1900)
}
ORDER = {"ngp": 1, "cic": 2, "tsc": 3}
MESHES = (16, 32, 64, 96, 128, 192, 256, 384, 512, 768, 1024)


def _estimate(name, entry, shape, mesh, scheme, interlace, ell, n_gal, n_ran, dk=0.01, k_max=0.0):
    return {"name": name, "entry": entry, "shape": shape, "mesh": mesh, "scheme": scheme, "interlace": interlace,
            "ell": ell, "n_gal": n_gal, "n_ran": n_ran, "dk": dk, "k_max": k_max}


def listed():
    return [
        # The smallest call: a first look at a small cube, result wanted at once.
        _estimate("cube32_cic", "measure", "cube", 32, "cic", False, 4, 2000, 10000),
        # One mock of a covariance run on a coarse mesh that fits L2, direct assignment.
        _estimate("mock128_direct", "direct", "cube", 128, "cic", False, 4, 1103417, 5517085, 0.01, 0.8),
        # A cone survey with FKP weights: one ordinary measurement, many in a row.
        _estimate("cone256_tsc_il", "assign", "cone", 256, "tsc", True, 4, 1000000, 5000000),
        # The same from the host's buffers: read from files, copied, measured, result on the host.
        _estimate("cone256_host", "host", "cone", 256, "tsc", True, 4, 1000000, 5000000),
        # The large survey, to k = 0.4: the library's headline workload.
        _estimate("survey512_tsc_il", "assign", "shell", 512, "tsc", True, 4, 10000000, 50000000, 0.01, 0.4),
        # The same survey with the hexacontatetrapole.
        _estimate("survey512_l6", "assign", "shell", 512, "tsc", True, 6, 10000000, 50000000, 0.01, 0.4),
        # Mock after mock against randoms that were deposited once.
        _estimate("survey512_shared", "cached", "shell", 512, "tsc", True, 4, 10000000, 50000000, 0.01, 0.4),
        # The paper's mock on its 1024^3 mesh, every shell up to Nyquist.
        _estimate("paper1024_cic", "assign", "cap", 1024, "cic", False, 4, 525000, 5250000),
        # Mocks of uneven sizes on mixed meshes in one graph launch.
        {"name": "batch24_mixed", "entry": "batch", "meshes": "128,192,256", "count": 24, "n_min": 200000,
         "n_max": 2000000, "correct": False},
        # The learned path: coarse measurements, then the network's correction of every shell.
        {"name": "learned128_x16", "entry": "batch", "meshes": "128", "count": 16, "n_min": 200000,
         "n_max": 2000000, "correct": True},
        # One full-batch gradient of the network's training.
        {"name": "mlp_grad_158k", "entry": "train", "rows": 158000},
        # The direct sum over galaxies of a small mock, the reference for aliasing.
        {"name": "sum_gal_64", "entry": "pairs", "mesh": 64, "ell": 4, "n_gal": 20000, "n_ran": 100000, "dk": 0.02},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(("assign",) * 5 + ("measure", "cached", "host", "direct", "batch", "train", "pairs"))
    if kind == "train":
        return {"entry": kind, "rows": _log_int(rng, 500, 200000)}
    if kind == "pairs":
        return {"entry": kind, "mesh": 2 * rng.randint(10, 32), "ell": rng.choice((0, 2, 4, 4, 6)),
                "n_gal": _log_int(rng, 300, 16000), "n_ran": _log_int(rng, 1000, 70000),
                "dk": round(rng.uniform(0.012, 0.04), 4)}
    if kind == "batch":
        meshes = rng.choice(("128", "64,128", "96,192", "128,192,256", "128,256", "192"))
        n_max = _log_int(rng, 30000, 2000000)
        return {"entry": kind, "meshes": meshes, "count": rng.randint(3, 24), "n_min": n_max // 10, "n_max": n_max,
                "correct": meshes == "128"}
    mesh = rng.choice(MESHES[:7] if kind == "direct" else MESHES)
    interlace = mesh <= 512 and rng.random() < 0.5 and not (kind == "direct" and mesh == 256)
    ell = rng.choice((0, 2, 4, 4, 4, 6)) if mesh <= 512 else rng.choice((0, 2, 4))
    shape = "cube" if mesh <= 64 else rng.choice(("cube", "cone", "shell", "cap"))
    n_gal = _log_int(rng, 1000, {16: 1e5, 32: 4e5, 64: 2e6}.get(mesh, 5e6 if mesh <= 512 else 8e5))
    nyquist = math.pi * mesh / BOXES[shape][1]
    scheme = rng.choice(("ngp", "cic", "cic", "tsc", "tsc", "tsc"))
    n_ran = int(n_gal * rng.uniform(1.5, 6.0))
    dk = round(rng.uniform(0.6, 4.0) * 2 * math.pi / BOXES[shape][1], 5)
    case = _estimate("", kind, shape, mesh, scheme, interlace, ell, n_gal, n_ran, dk, round(rng.uniform(0.4, 1.0) * nyquist, 5))
    del case["name"]
    return case


# --------------------------------------------------------------------------- catalogues

def _gen(seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed))
    return gen


def _rand(gen, *shape):
    return torch.rand(shape, generator=gen, device="cuda", dtype=torch.float64)


def _randn(gen, *shape):
    return torch.randn(shape, generator=gen, device="cuda", dtype=torch.float64)


def _clustered(gen, n, draw_points, sigma):
    """n points: half of them scattered about shared centres, half single (both drawn by draw_points)."""
    half = n // 2
    centres = draw_points(max(1, half // 20))
    near = centres[:, torch.randint(0, centres.shape[1], (half,), generator=gen, device="cuda")]
    near = near + sigma * _randn(gen, 3, half).clamp_(-4, 4)
    p = torch.cat([near, draw_points(n - half)], 1)
    return p[:, torch.randperm(n, generator=gen, device="cuda")]


def _catalogue(shape, n_gal, n_ran, seed):
    """(gal, ran): tuples of float32 device tensors (x, y, z, w, nbar), in random order."""
    gen = _gen(seed)
    lo, side = BOXES[shape]
    if shape == "cube":  # a clustered periodic cube, unit weights
        corner = torch.tensor(lo, dtype=torch.float64, device="cuda")[:, None]
        flat = lambda n: corner + side * _rand(gen, 3, n)  # noqa: E731
        gal, ran = corner + torch.remainder(_clustered(gen, n_gal, flat, 3.0) - corner, side), flat(n_ran)
        density, p_fkp = (lambda r: torch.full_like(r, n_gal / side ** 3)), 0.0
    elif shape == "shell":  # Poisson points of a clipped shell, unit weights
        share = [0.0]

        def flat(n):
            parts, have = [], 0
            while have < n:
                m = min(8_000_000, int(1.3 * (n - have)) + 1000)
                r = (600.0 ** 3 + _rand(gen, m) * (2000.0 ** 3 - 600.0 ** 3)) ** (1.0 / 3.0)
                d = _randn(gen, 3, m)
                p = d * (r / d.norm(dim=0))
                p = p[:, (p.abs() < 0.5 * side - 21.0).all(0)]
                share[0] = p.shape[1] / m
                parts.append(p)
                have += p.shape[1]
            return torch.cat(parts, 1)[:, :n]

        gal, ran = flat(n_gal), flat(n_ran)
        vol = share[0] * 4.0 / 3.0 * math.pi * (2000.0 ** 3 - 600.0 ** 3)
        density, p_fkp = (lambda r: torch.full_like(r, n_gal / vol)), 0.0
    else:  # clustered galaxies of a cone or cap, n(r) Gaussian, FKP weights
        mean, sd, r0, r1, p_fkp = (1200.0, 300.0, 300.0, 2100.0, 1e4) if shape == "cone" else (1500.0, 200.0, 1100.0, 1900.0, 2e4)
        cos_t = math.cos(math.radians(30.0)) if shape == "cone" else 1.0 - 7000.0 * (math.pi / 180.0) ** 2 / (2.0 * math.pi)
        axis = np.array([1.0, 1.0, 1.0]) / math.sqrt(3.0) if shape == "cone" else np.array([0.0, 0.0, 1.0])
        e1 = np.cross(axis, [1.0, 0.0, 0.0])
        e1 /= np.linalg.norm(e1)
        frame = torch.tensor(np.stack([e1, np.cross(axis, e1), axis], 1), device="cuda")
        a, b = (0.5 * (1.0 + math.erf((r - mean) / (sd * math.sqrt(2.0)))) for r in (r0, r1))

        def flat(n):
            r = mean + sd * math.sqrt(2.0) * torch.erfinv(2.0 * (a + (b - a) * _rand(gen, n)) - 1.0)
            ct = cos_t + (1.0 - cos_t) * _rand(gen, n)
            st, ph = (1.0 - ct * ct).clamp_min(0.0).sqrt(), 2.0 * math.pi * _rand(gen, n)
            return frame @ torch.stack([r * st * ph.cos(), r * st * ph.sin(), r * ct])

        gal, ran = _clustered(gen, n_gal, flat, 4.0), flat(n_ran)
        area = 2.0 * math.pi * (1.0 - cos_t) * sd * math.sqrt(2.0 * math.pi) * (b - a)
        density = lambda r: n_gal * torch.exp(-0.5 * ((r - mean) / sd) ** 2) / (area * r * r)  # noqa: E731

    def pack(p):
        p = p.to(torch.float32)
        for i in range(3):  # rounding must not carry a point onto the far face
            top = np.nextafter(np.float32(lo[i] + side), np.float32(-np.inf))
            p[i].clamp_(np.float32(lo[i]).item(), top.item())
        nbar = density(p.to(torch.float64).norm(dim=0))
        w = (1.0 / (1.0 + nbar * p_fkp)).to(torch.float32)
        return (p[0].contiguous(), p[1].contiguous(), p[2].contiguous(), w, nbar.to(torch.float32))

    return pack(gal), pack(ran)


def _batch_mocks(case, seed):
    rng = np.random.default_rng(seed)
    meshes = [int(m) for m in case["meshes"].split(",")]
    mocks = []
    for i in range(case["count"]):
        n = int(rng.integers(case["n_min"], case["n_max"] + 1))
        mesh = meshes[i % len(meshes)]
        mocks.append((mesh, n, _catalogue("cube", n, 5 * n, seed * 1000 + i)))
    return mocks


def _batch_bins(case):
    """Shells every 0.01 below the coarsest mesh's Nyquist frequency, the same for every mesh."""
    coarsest = min(int(m) for m in case["meshes"].split(","))
    return int(math.pi * coarsest / BOXES["cube"][1] / 0.01)


def _network(seed):
    """Parameters of a 5-64-64-64-3 network, uniform in +-1/sqrt(fan-in)."""
    rng = np.random.default_rng(seed + 17)
    parts = []
    for fan_in, fan_out in ((5, 64), (64, 64), (64, 64), (64, 3)):
        parts += [rng.uniform(-1, 1, fan_in * fan_out) / math.sqrt(fan_in), rng.uniform(-1, 1, fan_out) / math.sqrt(fan_in)]
    return np.concatenate(parts).astype(np.float32)


def _training_rows(case, seed):
    """Feature rows [k/k_N, ln(D/P_SN), P2/D, P4/D, P_SN/D] and residual targets of unit scale."""
    gen, n = _gen(seed), case["rows"]
    x = torch.empty((n, 5), dtype=torch.float32, device="cuda")
    x[:, 0] = torch.rand(n, generator=gen, device="cuda")
    x[:, 1] = 4.0 * torch.rand(n, generator=gen, device="cuda")
    x[:, 2:4] = 0.3 * torch.randn((n, 2), generator=gen, device="cuda")
    x[:, 4] = torch.exp(-x[:, 1])
    return x, torch.randn((n, 3), generator=gen, device="cuda")


# --------------------------------------------------------------------------- prepare, run

def _settings(case):
    lo, side = BOXES[case["shape"]]
    return dict(n_mesh=case["mesh"], box_min=lo, box_len=side, assign=case["scheme"], interlace=case["interlace"],
                ell_max=case["ell"], dk=case["dk"], k_max=case["k_max"] or None)


def prepare(case, seed):
    entry = case["entry"]
    if entry == "train":
        x, t = _training_rows(case, seed)
        return {"entry": entry, "net": ys.Mlp(_network(seed)), "x": x, "t": t,
                "grad": torch.empty(8899, device="cuda"), "sse": torch.empty(1, dtype=torch.float64, device="cuda")}
    if entry == "pairs":
        gal, ran = _catalogue("cube", case["n_gal"], case["n_ran"], seed)
        return {"entry": entry, "case": dict(case), "gal": gal, "ran": ran}
    if entry == "batch":
        mocks, nb = _batch_mocks(case, seed), _batch_bins(case)
        cfgs = [ys.make_config(mesh, *BOXES["cube"], assign="cic", dk=0.01, n_bins=nb, max_particles=6 * n) for mesh, n, _ in mocks]
        batch = ys.Batch(cfgs, lanes=8)
        rows = torch.zeros((len(mocks), batch.stride), dtype=torch.float64, device="cuda")
        state = {"entry": entry, "batch": batch, "gals": [c[0] for _, _, c in mocks], "rans": [c[1] for _, _, c in mocks],
                 "rows": rows, "n_bins": nb}
        if case["correct"]:
            state["net"], state["out"] = ys.Mlp(_network(seed)), torch.empty_like(rows)
            state["k_nyq"] = math.pi * mocks[0][0] / BOXES["cube"][1]
        return state
    gal, ran = _catalogue(case["shape"], case["n_gal"], case["n_ran"], seed)
    plan = ys.Plan(max_particles=case["n_gal"] + case["n_ran"], **_settings(case))
    state = {"entry": entry, "plan": plan, "gal": gal, "ran": ran}
    if entry == "host":
        state["pinned"] = [[a.cpu().pin_memory() for a in c] for c in (gal, ran)]
        state["gal"], state["ran"] = [[a.numpy() for a in c] for c in state["pinned"]]
    else:
        if entry == "direct":
            plan.set_direct_assign(True)
        if entry == "cached":
            plan.cache_randoms(ran)
        state["row"] = torch.zeros(plan.row_len, dtype=torch.float64, device="cuda")
    return state


def _result(res):
    out = {"k": res.k, "n_modes": res.n_modes, "p": np.stack([res.p0, res.p2, res.p4]).astype(np.float32),
           "sums": np.array([res.alpha, res.norm_I, res.shot_noise])}
    if res.p6 is not None:
        out["p6"] = res.p6.astype(np.float32)
    return out


def run(state):
    entry = state["entry"]
    if entry == "train":
        state["net"].gradient(state["x"], state["t"], state["grad"], state["sse"])
        return {"grad": state["grad"], "sse": state["sse"].float()}
    if entry == "pairs":
        c = state["case"]
        return _result(ys.sum_gal(c["mesh"], *BOXES["cube"], state["gal"], state["ran"], ell_max=c["ell"], dk=c["dk"]))
    if entry == "batch":
        nb, rows = state["n_bins"], state["rows"]
        state["batch"].run(state["gals"], state["rans"], rows)
        if "net" in state:
            state["net"].correct(rows, nb, state["k_nyq"], state["out"])
            rows = state["out"]
        return {"k": rows[:, :nb], "n_modes": rows[:, nb:2 * nb], "p": rows[:, 2 * nb:5 * nb].float(),
                "sums": rows[:, 5 * nb:5 * nb + 3]}
    plan = state["plan"]
    if entry == "host":
        return _result(plan.estimate_host(state["gal"], state["ran"]))
    if entry == "cached":
        plan.assign_cached(state["gal"])
    else:
        plan.assign(state["gal"], state["ran"])
    if entry == "measure":
        return _result(plan.measure())
    row, nb = state["row"], plan.n_bins
    plan.measure_async(row)
    out = {"k": row[:nb], "n_modes": row[nb:2 * nb], "p": row[2 * nb:5 * nb].float(), "sums": row[5 * nb:5 * nb + 3]}
    if plan.ell_max >= 6:
        out["p6"] = row[5 * nb + 5:].float()
    return out


def _estimate_work(mesh, order, meshes, ell, n_gal, n_ran, n_bins, ran_read=True):
    """Each catalogue read once (x, y, z, w, and nbar of the randoms), one row written; the stencil
    sums and the sum_l (2 l + 1) real transforms that multipoles up to l need."""
    n_ran = n_ran if ran_read else 0
    fields = sum(2 * l + 1 for l in range(0, ell + 1, 2))
    return {"bytes": 16 * n_gal + 20 * n_ran + 8 * (5 * n_bins + 5),
            "flops": meshes * (2 * order ** 3 * (n_gal + n_ran) + fields * 2.5 * mesh ** 3 * 3 * math.log2(mesh))}


def work(case):
    entry = case["entry"]
    if entry == "train":  # forward, the deltas and the weight gradients: three products per weight and row
        return {"bytes": 32 * case["rows"] + 4 * 8899, "flops": 3 * 2 * 8704 * case["rows"]}
    if entry == "pairs":  # per mode and point: the phase, its cosine and sine, mu, and two sums per multipole
        modes = 2.0 / 3.0 * math.pi * (case["mesh"] / 2) ** 3
        n = case["n_gal"] + case["n_ran"]
        return {"bytes": 20 * n, "flops": modes * n * (5 + 2 + 6 + 4 * (case["ell"] // 2 + 1))}
    if entry == "batch":
        meshes = [int(m) for m in case["meshes"].split(",")]
        n, total = (case["n_min"] + case["n_max"]) // 2, {"bytes": 0, "flops": 0}
        for i in range(case["count"]):
            w = _estimate_work(meshes[i % len(meshes)], 2, 1, 4, n, 5 * n, _batch_bins(case))
            total = {k: total[k] + w[k] for k in total}
        return total
    n_bins = math.ceil((case["k_max"] or math.pi * case["mesh"] / BOXES[case["shape"]][1]) / case["dk"] - 1e-9)
    return _estimate_work(case["mesh"], ORDER[case["scheme"]], 2 if case["interlace"] else 1, case["ell"],
                          case["n_gal"], case["n_ran"], n_bins, entry != "cached")


# --------------------------------------------------------------------------- 64 bits

def _deposit(mesh, cat, scale, n, lo, side, order, shift):
    """mesh += scale w W(u - node) in 64 bits, u = (x - lo) n / side - shift."""
    for s in range(0, cat[0].shape[0], 4_000_000):
        w = cat[3][s:s + 4_000_000].double() * scale
        axes = []
        for a in range(3):
            u = (cat[a][s:s + 4_000_000].double() - lo[a]) * (n / side) - shift
            i = torch.floor(u) if order == 2 else torch.floor(u + 0.5)
            d = u - i
            st = ([(i, None)] if order == 1 else [(i, 1.0 - d), (i + 1, d)] if order == 2 else
                  [(i - 1, 0.5 * (0.5 - d) ** 2), (i, 0.75 - d * d), (i + 1, 0.5 * (0.5 + d) ** 2)])
            axes.append([(torch.remainder(j, n).long(), v) for j, v in st])
        for ix, wx in axes[0]:
            for iy, wy in axes[1]:
                for iz, wz in axes[2]:
                    mesh.index_add_(0, (ix * n + iy) * n + iz, w if wx is None else w * wx * wy * wz)


def _monomials(d):
    for a in range(d + 1):
        for b in range(d + 1 - a):
            c = d - a - b
            yield math.factorial(d) // (math.factorial(a) * math.factorial(b) * math.factorial(c)), a, b, c


def _exact_estimate(gal, ran, lo, side, n, scheme, interlace, ell, dk, n_bins):
    order = ORDER[scheme]
    wg, wr, nb = gal[3].double(), ran[3].double(), ran[4].double()
    alpha = float(wg.sum() / wr.sum())
    norm, shot = alpha * float((wr * wr * nb).sum()), float((wg * wg).sum()) + alpha ** 2 * float((wr * wr).sum())
    f = torch.fft.fftfreq(n, 1.0 / n, device="cuda", dtype=torch.float64)
    h = torch.arange(n // 2 + 1, device="cuda", dtype=torch.float64)
    k = (f[:, None, None], f[None, :, None], h[None, None, :])
    total = {}
    for j in range(2 if interlace else 1):
        mesh = torch.zeros(n ** 3, dtype=torch.float64, device="cuda")
        _deposit(mesh, gal, 1.0, n, lo, side, order, 0.5 * j)
        _deposit(mesh, ran, -alpha, n, lo, side, order, 0.5 * j)
        mesh = mesh.view(n, n, n)
        r = [(lo[a] + (torch.arange(n, device="cuda", dtype=torch.float64) + 0.5 * j) * (side / n)) for a in range(3)]
        r = (r[0][:, None, None], r[1][None, :, None], r[2][None, None, :])
        r2 = r[0] ** 2 + r[1] ** 2 + r[2] ** 2
        inv = torch.where(r2 > 0, 1.0 / r2, torch.zeros_like(r2))
        del r2
        for d in range(0, ell + 1, 2):
            acc = torch.zeros((n, n, n // 2 + 1), dtype=torch.complex128, device="cuda")
            for coef, a, b, c in _monomials(d):
                t = torch.fft.rfftn(mesh * (r[0] ** a) * (r[1] ** b) * (r[2] ** c))
                acc += t.mul_(coef * k[0] ** a).mul_(k[1] ** b).mul_(k[2] ** c)
                del t
            if interlace:
                for q in k if j == 1 else ():
                    acc *= torch.exp(-1j * math.pi / n * q)
                acc *= 0.5
            total[d] = total[d] + acc if j else acc
            del acc
            mesh = mesh * inv
        del mesh, inv
    n2 = (k[0] ** 2 + k[1] ** 2 + k[2] ** 2)
    keep = (n2 > 0) & (n2 < (n // 2) ** 2)
    n2 = n2[keep].long()
    window = torch.ones((n, n, n // 2 + 1), dtype=torch.float64, device="cuda")
    for q in k:
        x = q * (math.pi / n)
        window *= torch.where(x == 0, torch.ones_like(x), torch.sin(x) / torch.where(x == 0, torch.ones_like(x), x)) ** (2 * order)
    weight = ((1.0 + ((k[2] > 0) & (k[2] < n // 2)).double()) / window)[keep]
    size = (n // 2) ** 2
    kmag = 2.0 * math.pi / side * torch.arange(size, device="cuda", dtype=torch.float64).sqrt()
    shell = torch.floor(kmag / dk)
    ok = (shell < n_bins) & (kmag < 2.0 * math.pi / side * n / 2.0) & (kmag > 0)

    def to_shells(v):
        by_n2 = torch.zeros(size, dtype=torch.float64, device="cuda").index_add_(0, n2, v)
        return torch.zeros(n_bins, dtype=torch.float64, device="cuda").index_add_(0, shell[ok].long(), by_n2[ok])

    a0 = total[0][keep]
    count = to_shells((1.0 + ((k[2] > 0) & (k[2] < n // 2)).double()).expand(n, n, n // 2 + 1)[keep])
    m = {}
    for d in total:
        ad = total[d][keep]
        m[d] = to_shells(weight * (a0.real * ad.real + a0.imag * ad.imag) / n2.double() ** (d // 2)) / count
    nan = torch.full_like(count, math.nan)
    p0, p2, p4 = (m[0] - shot) / norm, nan, nan
    if ell >= 2:
        p2 = 2.5 / norm * (3.0 * m[2] - m[0])
    if ell >= 4:
        p4 = 1.125 / norm * (35.0 * m[4] - 30.0 * m[2] + 3.0 * m[0])
    out = {"k": None, "n_modes": None, "p": torch.stack([p0, p2, p4]),
           "sums": torch.tensor([alpha, norm, shot / norm], dtype=torch.float64)}
    if ell >= 6:
        out["p6"] = 0.8125 / norm * (231.0 * m[6] - 315.0 * m[4] + 105.0 * m[2] - 5.0 * m[0])
    return out, count


def _bf16(params):
    return torch.from_numpy(params).to(torch.bfloat16).double().cuda()


def _layers(params):
    at, out = 0, []
    for fan_in, fan_out in ((5, 64), (64, 64), (64, 64), (64, 3)):
        w = params[at:at + fan_in * fan_out].view(fan_out, fan_in)
        at += fan_in * fan_out
        out.append((w, params[at:at + fan_out]))
        at += fan_out
    return out


def _apply(params, x):
    layers = _layers(params)
    for i, (w, b) in enumerate(layers):
        x = x @ w.T + b
        if i < len(layers) - 1:
            x = 0.5 * x * (1.0 + torch.erf(x / math.sqrt(2.0)))
    return x


def _exact_pairs(gal, ran, lo, side, n, ell, dk):
    """A_n(k) by factored phases: for each m_x the sums over (m_y, m_z) are matrix products."""
    wg, wr, nb = gal[3].double(), ran[3].double(), ran[4].double()
    alpha = float(wg.sum() / wr.sum())
    norm, shot = alpha * float((wr * wr * nb).sum()), float((wg * wg).sum()) + alpha ** 2 * float((wr * wr).sum())
    p = [torch.cat([gal[a], ran[a]]).double() for a in range(3)]
    w = torch.cat([wg, -alpha * wr])
    r = torch.stack(p)
    rhat = r / r.norm(dim=0)
    n_bins = math.ceil(math.pi * n / side / dk - 1e-9)
    m = torch.arange(-(n // 2), n // 2, device="cuda", dtype=torch.float64)
    mz = torch.arange(0, n // 2 + 1, device="cuda", dtype=torch.float64)
    phase = lambda q, a: torch.exp(-2j * math.pi * q[:, None] * ((p[a] - lo[a]) / side)[None])  # noqa: E731
    ey, ez = phase(m, 1), phase(mz, 2)
    shells = {d: torch.zeros(n_bins, dtype=torch.float64, device="cuda") for d in range(0, ell + 1, 2)}
    count = torch.zeros(n_bins, dtype=torch.float64, device="cuda")
    kf = 2.0 * math.pi / side
    for mx in m.tolist():
        ex = torch.exp(-2j * math.pi * mx * ((p[0] - lo[0]) / side)) * w
        n2 = mx * mx + m[:, None] ** 2 + mz[None] ** 2
        kmag = kf * n2.sqrt()
        b = torch.floor(kmag / dk)
        ok = (n2 > 0) & (kmag < kf * n / 2.0) & (b < n_bins)
        herm = 1.0 + ((mz > 0) & (mz < n // 2)).double()[None].expand_as(n2)
        count.index_add_(0, b[ok].long(), herm[ok])
        amp = {}
        for d in shells:
            acc = torch.zeros_like(n2, dtype=torch.complex128)
            for coef, a, bb, c in _monomials(d):
                if mx == 0 and a:
                    continue
                v = ex * (coef * mx ** a) * rhat[0] ** a * rhat[1] ** bb * rhat[2] ** c
                acc += ((ey * v[None]) @ ez.T) * m[:, None] ** bb * mz[None] ** c
            amp[d] = acc
            v = herm * (amp[0].real * acc.real + amp[0].imag * acc.imag) / n2.clamp_min(1.0) ** (d // 2)
            shells[d].index_add_(0, b[ok].long(), v[ok])
    q = {d: v / count for d, v in shells.items()}
    nan = torch.full_like(count, math.nan)
    out = {"k": None, "n_modes": None,
           "p": torch.stack([(q[0] - shot) / norm, 2.5 / norm * (3.0 * q[2] - q[0]) if ell >= 2 else nan,
                             1.125 / norm * (35.0 * q[4] - 30.0 * q[2] + 3.0 * q[0]) if ell >= 4 else nan]),
           "sums": torch.tensor([alpha, norm, shot / norm], dtype=torch.float64)}
    if ell >= 6:
        out["p6"] = 0.8125 / norm * (231.0 * q[6] - 315.0 * q[4] + 105.0 * q[2] - 5.0 * q[0])
    return out


def exact(case, seed):
    entry = case["entry"]
    if entry == "train":
        x, t = _training_rows(case, seed)
        params = _bf16(_network(seed)).requires_grad_()
        err = _apply(params, x.double()) - t.double()
        (err.square().sum() / err.numel()).backward()
        return {"grad": params.grad, "sse": err.detach().square().sum().view(1)}
    if entry == "pairs":
        gal, ran = _catalogue("cube", case["n_gal"], case["n_ran"], seed)
        return _exact_pairs(gal, ran, *BOXES["cube"], case["mesh"], case["ell"], case["dk"])
    if entry == "batch":
        nb, params = _batch_bins(case), _bf16(_network(seed))
        ps, sums = [], []
        for mesh, _, (gal, ran) in _batch_mocks(case, seed):
            out, count = _exact_estimate(gal, ran, *BOXES["cube"], mesh, "cic", False, 4, 0.01, nb)
            p = out["p"]
            if case["correct"]:  # shells with modes, finite multipoles and D > 0 are corrected
                shot = float(out["sums"][2])
                d = p[0] + shot
                # the mean |k| of a shell's modes, from the integer lattice
                kf, half = 2.0 * math.pi / BOXES["cube"][1], mesh // 2
                f = torch.fft.fftfreq(mesh, 1.0 / mesh, device="cuda", dtype=torch.float64)
                n2 = f[:, None, None] ** 2 + f[None, :, None] ** 2 + f[None, None, :] ** 2
                n2 = n2[(n2 > 0) & (n2 < half * half)]
                km = kf * n2.sqrt()
                b = torch.floor(km / 0.01).long()
                ok = b < nb
                z = torch.zeros(nb, dtype=torch.float64, device="cuda")
                kbar = z.clone().index_add_(0, b[ok], km[ok]) / z.index_add_(0, b[ok], torch.ones_like(km[ok]))
                use = (count > 0) & (d > 0)
                x = torch.stack([kbar / (math.pi * mesh / BOXES["cube"][1]), torch.log(d / shot), p[1] / d, p[2] / d, shot / d], 1)
                p = torch.where(use[None], p + d[None] * _apply(params, x).T, p)
            ps.append(p.reshape(-1))
            sums.append(out["sums"])
        return {"k": None, "n_modes": None, "p": torch.stack(ps), "sums": torch.stack(sums)}
    gal, ran = _catalogue(case["shape"], case["n_gal"], case["n_ran"], seed)
    lo, side = BOXES[case["shape"]]
    n_bins = math.ceil((case["k_max"] or math.pi * case["mesh"] / side) / case["dk"] - 1e-9)
    out, _ = _exact_estimate(gal, ran, lo, side, case["mesh"], case["scheme"], case["interlace"], case["ell"],
                             case["dk"], n_bins)
    if entry not in ("measure", "host"):  # rows hold the multipoles one after another
        out["p"] = out["p"].reshape(-1)
    return out
