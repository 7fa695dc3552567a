"""Performance cases: the calls a program makes through the package's public
entry points, over the range of sizes it makes them with.

Kinds of case:
  step      one or more kick-drift-kick steps of a galaxy (tree build, tree or
            direct gravity, kernel sizes, density, hydro force) and the state
            read back: what every global step of a simulation runs
  gravity   particles handed over, self-gravity, forces read back: the library
            as the force routine of another integrator
  sn        plain CFL-limited integration of one supernova region (the training
            signal of the surrogate, and its fallback)
  voxelise  supernova regions onto grids: the surrogate's input
  remap     particles of supernova regions redrawn from predicted grids, and
            the sort and tree build that follow it
  forward   the U-Net over a batch of regions: the surrogate's inference
  train     one training step of the U-Net (forward, loss, backward, Adam)

Inputs are drawn on the GPU from the seed, with the distributions of the
package's initial conditions (Plummer sphere, exponential disk in a static
halo, turbulent log-normal regions).
"""
import math

import torch

from paper_2510_23330_gb300 import galnb, ics, surrogate

DEV = "cuda"
SIDE = 60.0                       # pc, edge of a supernova region
MODES = {"tree": galnb.GNB_GRAV_TREE, "direct": galnb.GNB_GRAV_DIRECT, "none": galnb.GNB_GRAV_NONE}
STEP_FIELDS = ("X", "Y", "Z", "VX", "VY", "VZ", "U", "AX", "AY", "AZ", "POT", "DUDT", "RHO", "H2")
STAR_FIELDS = ("X", "Y", "Z", "VX", "VY", "VZ", "AX", "AY", "AZ", "POT")
GRAV_FIELDS = ("AX", "AY", "AZ", "POT")
SN_FIELDS = ("X", "Y", "Z", "VX", "VY", "VZ", "U", "AX", "AY", "AZ", "DUDT", "RHO", "H2")
REMAP_FIELDS = ("X", "Y", "Z", "VX", "VY", "VZ", "U", "KEY", "ORDER")
TORCH_DTYPE = {"X": torch.float64, "Y": torch.float64, "Z": torch.float64, "H2": torch.float64,
               "KEY": torch.int64, "ORDER": torch.int64}


def listed():
    return [
        # the tiny model of the tests and the examples: launches and host waits count
        {"name": "step_plummer_8k", "kind": "step", "model": "plummer", "n": 8192, "gas": 0.5, "n_group": 64,
         "gravity": "tree", "multipole": 1, "pressure": False, "steps": 1},
        # a development-size galaxy with an odd count and the default group size
        {"name": "step_disk_150k", "kind": "step", "model": "disk", "n": 150001, "gas": 0.2, "n_group": 64,
         "gravity": "tree", "multipole": 1, "pressure": False, "steps": 1},
        # the 2^20 disk at the group size the tuner picked for it
        {"name": "step_disk_2p20", "kind": "step", "model": "disk", "n": 1 << 20, "gas": 0.2, "n_group": 128,
         "gravity": "tree", "multipole": 1, "pressure": False, "steps": 1},
        # the 2^24 disk, the largest single-GPU model, at its tuned group size
        {"name": "step_disk_2p24", "kind": "step", "model": "disk", "n": 1 << 24, "gas": 0.1, "n_group": 256,
         "gravity": "tree", "multipole": 1, "pressure": False, "steps": 1},
        # a star cluster with per-particle softening in another code's integrator: monopole tree, default groups
        {"name": "gravity_stars_300k", "kind": "gravity", "n": 300007, "n_group": 64, "gravity": "tree",
         "multipole": 0, "eps": "mixed"},
        # exact forces of a small system (collisional work, checks of the tree)
        {"name": "gravity_direct_20k", "kind": "gravity", "n": 20011, "n_group": 64, "gravity": "direct",
         "multipole": 1, "eps": "uniform"},
        # one region of the training set
        {"name": "sn_plain_100k", "kind": "sn", "n": 100000, "pressure": False, "steps": 12},
        # the smallest regions of the coupled batch, pressure-energy SPH
        {"name": "sn_plain_20k_pressure", "kind": "sn", "n": 20011, "pressure": True, "steps": 12},
        # a ragged batch of regions on their way into the network
        {"name": "voxelise_64", "kind": "voxelise", "nreg": 64, "n_min": 20000, "n_max": 300000, "grid": 64},
        # and back to particles
        {"name": "remap_64", "kind": "remap", "nreg": 64, "n_min": 20000, "n_max": 300000, "grid": 64, "sweeps": 8},
        # inference over a batch of regions
        {"name": "unet_forward_32", "kind": "forward", "batch": 32, "grid": 64, "base": 16, "levels": 4},
        # training at batch size 1, as the network is trained
        {"name": "unet_train_1", "kind": "train", "batch": 1, "grid": 64, "base": 16, "levels": 4},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step", "step", "step", "gravity", "gravity", "sn", "sn", "voxelise", "remap", "forward",
                       "train"])
    if kind == "step":
        n = _log_int(rng, 4096, 4 << 20)
        return {"kind": kind, "model": rng.choice(["plummer", "disk"]), "n": n,
                "gas": rng.choice([0.0, 0.1, 0.2, 0.5]),
                "n_group": rng.choice([32, 64, 128, 192, 256]), "gravity": "tree",
                "multipole": rng.choice([0, 1, 1]), "pressure": rng.random() < 0.3, "steps": rng.choice([1, 2, 3])}
    if kind == "gravity":
        direct = rng.random() < 0.5
        return {"kind": kind, "n": _log_int(rng, 500, 60000 if direct else 1000000),
                "n_group": rng.choice([32, 64, 128, 256]), "gravity": "direct" if direct else "tree",
                "multipole": rng.choice([0, 1]), "eps": rng.choice(["uniform", "mixed"])}
    if kind == "sn":
        return {"kind": kind, "n": _log_int(rng, 5000, 300000), "pressure": rng.random() < 0.5,
                "steps": rng.randint(3, 12)}
    if kind in ("voxelise", "remap"):
        lo = _log_int(rng, 5000, 40000)
        c = {"kind": kind, "nreg": _log_int(rng, 1, 32), "n_min": lo, "n_max": _log_int(rng, lo, 200000),
             "grid": rng.choice([32, 64, 64])}
        if kind == "remap":
            c["sweeps"] = rng.randint(2, 8)
        return c
    if kind == "forward":
        return {"kind": kind, "batch": _log_int(rng, 1, 48), "grid": rng.choice([16, 24, 32, 40, 48, 64]),
                "base": 16, "levels": rng.choice([3, 4])}
    return {"kind": "train", "batch": rng.randint(1, 4), "grid": rng.choice([16, 24, 32, 40, 48]), "base": 16,
            "levels": rng.choice([3, 4])}


# ------------------------------------------------------------------ particles
def _gen(seed, salt=0):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed) * 1000003 + salt)
    return g


def _u(g, n):
    return torch.rand(n, generator=g, device=DEV, dtype=torch.float64)


def _iso(g, n):
    cz = 2.0 * _u(g, n) - 1.0
    ph = 2.0 * math.pi * _u(g, n)
    s = torch.sqrt(1.0 - cz * cz)
    return torch.stack([s * torch.cos(ph), s * torch.sin(ph), cz])


def _pack(x, v, m, eps, u, gas):
    n = x.shape[1]
    f = torch.float32
    return {"id": torch.arange(n, device=DEV, dtype=torch.int64), "type": gas.to(torch.uint8).contiguous(),
            "x": x[0].contiguous(), "y": x[1].contiguous(), "z": x[2].contiguous(),
            "vx": v[0].to(f).contiguous(), "vy": v[1].to(f).contiguous(), "vz": v[2].to(f).contiguous(),
            "m": m.to(f).contiguous(), "eps": eps.to(f).contiguous(), "u": u.to(f).contiguous()}


def _full(n, v):
    return torch.full((n,), float(v), device=DEV, dtype=torch.float64)


def _plummer(n, seed, n_gas, u_gas=0.05, eps="uniform"):
    """Plummer sphere, G = M = a = 1, radii up to 100; gas last."""
    g = _gen(seed)
    x1 = _u(g, n) * (1.0 + 1e-4) ** -1.5 + 1e-12
    r = 1.0 / torch.sqrt(x1 ** (-2.0 / 3.0) - 1.0)
    pos = _iso(g, n) * r
    # speed over escape speed from q^2 (1 - q^2)^(7/2), by the inverse of its tabulated integral
    q = torch.linspace(0.0, 1.0, 4097, device=DEV, dtype=torch.float64)
    w = q * q * (1.0 - q * q).clamp_min(0.0) ** 3.5
    cdf = torch.cat([_full(1, 0.0), torch.cumsum(0.5 * (w[1:] + w[:-1]), 0)])
    cdf = cdf / cdf[-1]
    t = _u(g, n)
    k = torch.searchsorted(cdf, t).clamp(1, 4096)
    qq = q[k - 1] + (t - cdf[k - 1]) / (cdf[k] - cdf[k - 1]).clamp_min(1e-300) * (q[1] - q[0])
    vel = _iso(g, n) * (qq * math.sqrt(2.0) * (1.0 + r * r) ** -0.25)
    gas = torch.arange(n, device=DEV) >= n - n_gas
    e = _full(n, 0.01) if eps == "uniform" else 0.005 * 10.0 ** _u(g, n)
    return _pack(pos, vel, _full(n, 1.0 / n), e, torch.where(gas, u_gas, 0.0), gas)


def _disk(n, seed, gas_frac):
    """Exponential stellar and gas disks in the static NFW halo of the package's disk model; stars first."""
    g = _gen(seed)
    n_gas = int(round(gas_frac * n))
    gas = torch.arange(n, device=DEV) >= n - n_gas
    rd = torch.where(gas, 2.0, 1.0).to(torch.float64)
    R = -rd * torch.log(_u(g, n).clamp_min(1e-300) * _u(g, n).clamp_min(1e-300))
    ph = 2.0 * math.pi * _u(g, n)
    z = 0.1 * torch.atanh((2.0 * _u(g, n) - 1.0).clamp(-1.0 + 1e-12, 1.0 - 1e-12))
    pos = torch.stack([R * torch.cos(ph), R * torch.sin(ph), z])
    r = torch.sqrt(R * R + z * z)
    rank = torch.empty(n, device=DEV, dtype=torch.float64)
    rank[torch.argsort(r)] = torch.arange(1, n + 1, device=DEV, dtype=torch.float64)
    s = r / ics.NFW_RS
    menc = rank / n + ics.NFW_MS * (torch.log1p(s) - s / (1.0 + s))
    vc = torch.sqrt(menc / r.clamp_min(1e-6)) * (R / r.clamp_min(1e-12))
    vel = torch.stack([-torch.sin(ph), torch.cos(ph), torch.zeros_like(ph)]) * vc
    sig = torch.where(gas, 0.0, 0.1 * vc)
    vel = vel + torch.randn((3, n), generator=g, device=DEV, dtype=torch.float64) * sig
    u = torch.where(gas, torch.exp(math.log(1e-3) + math.log(1e2) * _u(g, n)), 0.0)
    return _pack(pos, vel, _full(n, 1.0 / n), _full(n, 0.01), u, gas)


def _grf(g, ng, ncomp, solenoidal=False):
    """Gaussian random fields with P(k) ~ k^(-11/3) on an ng^3 grid, zero mean, unit variance."""
    k = torch.fft.fftfreq(ng, device=DEV, dtype=torch.float64) * ng
    kz = torch.fft.rfftfreq(ng, device=DEV, dtype=torch.float64) * ng
    K = torch.stack(torch.meshgrid(k, k, kz, indexing="ij"))
    k2 = (K * K).sum(0)
    safe = torch.where(k2 > 0, k2, 1.0)
    amp = torch.where(k2 > 0, safe ** (-11.0 / 12.0), 0.0)
    ph = torch.randn((2, ncomp) + k2.shape, generator=g, device=DEV, dtype=torch.float64)
    f = torch.complex(ph[0], ph[1]) * amp
    if solenoidal:
        f = f - K * (K * f).sum(0) / safe
    f = torch.fft.irfftn(f, s=(ng, ng, ng), dim=(1, 2, 3))
    f = f - f.mean(dim=(1, 2, 3), keepdim=True)
    return f / f.std(dim=(1, 2, 3), keepdim=True)


def _region(n, seed, salt=0, ng=64):
    """Positions and velocities of one turbulent region centred on the origin."""
    g = _gen(seed, salt)
    f = _grf(g, ng, 1)[0].reshape(-1)
    cell = torch.multinomial(torch.exp(f - 0.5), n, replacement=True, generator=g)
    ijk = torch.stack([cell // (ng * ng), cell // ng % ng, cell % ng]).to(torch.float64)
    pos = (ijk + torch.rand((3, n), generator=g, device=DEV, dtype=torch.float64)) * (SIDE / ng) - 0.5 * SIDE
    v = _grf(g, ng, 3, solenoidal=True).reshape(3, -1)[:, cell]
    return pos, v * (10.0 / torch.sqrt((v * v).sum(0).mean()))


def _sn_region(n, seed):
    """One region just after the explosion: 10^51 erg in the 64 gas particles nearest to its centre."""
    pos, v = _region(n, seed)
    u = _full(n, 100.0 / ics.T_PER_U)
    d = torch.sqrt((pos * pos).sum(0))
    near = torch.topk(d, 64, largest=False)
    q = near.values / near.values.max()
    w = torch.where(q <= 0.5, 1 - 6 * q ** 2 + 6 * q ** 3, 2 * (1 - q) ** 3)
    u[near.indices] += ics.E_SN_CODE * w / w.sum()
    return _pack(pos, v, _full(n, 1.0), _full(n, 0.1), u, torch.ones(n, device=DEV, dtype=torch.bool))


def _sizes(case):
    """Member counts, log-uniform between the smallest and the largest region."""
    k, lo, hi = case["nreg"], case["n_min"], case["n_max"]
    return [int(lo * (hi / lo) ** ((r + 0.5) / k)) for r in range(k)]


def _centres(case):
    return [(3.0 * SIDE * (r % 16), 3.0 * SIDE * (r // 16), 0.0) for r in range(case["nreg"])]


def _regions(case, seed):
    """The regions of a batch, 180 pc apart in one particle set."""
    P, V = [], []
    for r, (n, c) in enumerate(zip(_sizes(case), _centres(case))):
        pos, v = _region(n, seed, 1 + r)
        P.append(pos + torch.tensor(c, device=DEV, dtype=torch.float64)[:, None])
        V.append(v)
    pos, v = torch.cat(P, 1), torch.cat(V, 1)
    n = pos.shape[1]
    u = (30.0 + 300.0 * _u(_gen(seed, 999), n)) / ics.T_PER_U
    return _pack(pos, v, _full(n, 1.0), _full(n, 0.1), u, torch.ones(n, device=DEV, dtype=torch.bool))


def _prediction(case, seed):
    """Grids like the network's: log density, log temperature and velocity in its standardised units."""
    G, out = case["grid"], []
    for r in range(case["nreg"]):
        f = _grf(_gen(seed, 5000 + r), G, 5).reshape(5, -1)
        out.append(torch.stack([0.43 * f[0] - 0.2, 0.4 * f[1] + 0.3, 0.5 * f[2], 0.5 * f[3], 0.5 * f[4]], 1))
    return torch.stack(out).to(torch.float32).contiguous()


def _particles(case, seed):
    if case["kind"] == "step":
        if case["model"] == "plummer":
            return _plummer(case["n"], seed, int(round(case["gas"] * case["n"])))
        return _disk(case["n"], seed, case["gas"])
    if case["kind"] == "gravity":
        return _plummer(case["n"], seed, 0, eps=case["eps"])
    if case["kind"] == "sn":
        return _sn_region(case["n"], seed)
    return _regions(case, seed)


def _grids(case, seed):
    """Network inputs and targets: correlated standardised fields."""
    B, G = case["batch"], case["grid"]
    f = [torch.stack([_grf(_gen(seed, 7000 + 2 * b + s), G, 5) for b in range(B)]) for s in range(2)]
    f = [(0.5 * t).permute(0, 2, 3, 4, 1).to(torch.float32).contiguous() for t in f]
    return f[0], (0.8 * f[0] + 0.3 * f[1]).contiguous()


def _net(case, seed):
    net = galnb.UNet(5, 5, case["base"], case["levels"], case["grid"])
    w = surrogate.he_init(5, 5, case["base"], case["levels"], seed=seed % (1 << 31))
    net.set_params(w)
    return net, w


def _halo(case):
    return {"nfw_ms": ics.NFW_MS, "nfw_rs": ics.NFW_RS} if case.get("model") == "disk" else {}


def _buffers(fields, n):
    return {k: torch.empty(n, device=DEV, dtype=TORCH_DTYPE.get(k, torch.float32)) for k in fields}


# ------------------------------------------------------------------ the cases
def prepare(case, seed):
    kind = case["kind"]
    if kind in ("forward", "train"):
        net, _ = _net(case, seed)
        x, t = _grids(case, seed)
        s = {"case": case, "net": net, "x": x, "t": t}
        if kind == "forward":
            s["y"] = torch.empty_like(x)
        else:
            s["grads"] = torch.empty(net.num_params(), device=DEV)
            s["params"] = torch.empty(net.num_params(), device=DEV)
        torch.cuda.synchronize()
        return s
    p = _particles(case, seed)
    n = p["x"].shape[0]
    torch.cuda.synchronize()
    s = {"case": case, "p": p}
    if kind == "step":
        c = galnb.Context(n_group=case["n_group"], multipole=case["multipole"],
                          sph_variant=1 if case["pressure"] else 0, **_halo(case))
        c.set_particles(p)
        c.compute_forces(MODES[case["gravity"]])
        s["out"] = _buffers(STEP_FIELDS if case["gas"] else STAR_FIELDS, n)
    elif kind == "gravity":
        c = galnb.Context(n_group=case["n_group"], multipole=case["multipole"])
        s["out"] = _buffers(GRAV_FIELDS, n)
    elif kind == "sn":
        c = galnb.Context(sph_variant=1 if case["pressure"] else 0)
        s["out"] = _buffers(SN_FIELDS, n)
    else:
        c = galnb.Context()
        c.set_particles(p)
        G = case["grid"]
        s["centres"] = galnb._centers(_centres(case))
        if kind == "voxelise":
            c.compute_sph_density()
            s["out"] = torch.empty((case["nreg"], G ** 3, 5), device=DEV)
        else:
            c.build_tree()
            s["pred"] = _prediction(case, seed)
            s["seed"] = int(seed)
            s["out"] = _buffers(REMAP_FIELDS, n)
    s["ctx"] = c
    torch.cuda.synchronize()
    return s


DT = 1e-3  # global step of the galaxy models


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "step":
        c = s["ctx"]
        c.step_kdk(DT, case["steps"], MODES[case["gravity"]])
        return c.get_fields(s["out"])
    if kind == "gravity":
        c = s["ctx"]
        c.set_particles(s["p"])
        c.compute_gravity(MODES[case["gravity"]])
        return c.get_fields(s["out"])
    if kind == "sn":
        c = s["ctx"]
        c.set_particles(s["p"])
        t, steps = c.integrate_cfl(ics.T_SN_END, 0.3, max_steps=case["steps"], mode=galnb.GNB_GRAV_NONE)
        return dict(c.get_fields(s["out"]), steps=steps, t=t)
    if kind == "voxelise":
        c = s["ctx"]
        c._chk(galnb.gnb_voxelise(c.h, case["nreg"], s["centres"][1], SIDE, case["grid"], s["out"].data_ptr(), 1))
        return s["out"]
    if kind == "remap":
        c = s["ctx"]
        c._chk(galnb.gnb_remap_regions(c.h, case["nreg"], s["centres"][1], SIDE, case["grid"], s["pred"].data_ptr(),
                                       s["seed"], case["sweeps"], 1))
        c.build_tree()
        return c.get_fields(s["out"])
    net = s["net"]
    if kind == "forward":
        return net.forward(s["x"], out=s["y"])
    loss = net.train_step(s["x"], s["t"], 1e-3)
    net._chk(galnb.gnb_unet_get_grads(net.h, s["grads"].data_ptr(), 1), "get_grads")
    net._chk(galnb.gnb_unet_get_params(net.h, s["params"].data_ptr(), 1), "get_params")
    return {"loss": loss, "grads": s["grads"], "params": s["params"]}


def _net_shape(case):
    """(kind, cin, cout, level) of the network's layers, in parameter order."""
    b, L, c, out = case["base"], case["levels"], 5, []
    for l in range(L):
        out += [("conv", c, b << l, l), ("conv", b << l, b << l, l)]
        c = b << l
    for l in range(L - 2, -1, -1):
        out += [("up", b << (l + 1), b << l, l), ("conv", 2 * (b << l), b << l, l), ("conv", b << l, b << l, l)]
    return out + [("head", b, 5, 0)]


def work(case):
    kind = case["kind"]
    if kind in ("forward", "train"):
        v0 = case["batch"] * case["grid"] ** 3
        flops = params = 0
        for k, ci, co, l in _net_shape(case):
            # a transposed convolution applies one of its taps to each fine voxel
            flops += 2 * (27 if k == "conv" else 1) * ci * co * (v0 >> (3 * l))
            params += {"conv": 27, "up": 8, "head": 1}[k] * ci * co + co
        if kind == "forward":
            return {"bytes": 4 * (10 * v0 + params), "flops": flops}
        return {"bytes": 4 * (10 * v0 + 9 * params), "flops": 3 * flops}
    if kind in ("voxelise", "remap"):
        n, nv = sum(_sizes(case)), case["nreg"] * case["grid"] ** 3
        if kind == "voxelise":
            # every voxel sums over the particles whose support covers it, 64 on average
            return {"bytes": 52 * n + 20 * nv, "flops": 64 * 20 * nv}
        # read and write each particle, the grid, its three sets of line sums; then the sort and the tree
        return {"bytes": n * (60 + 36 + 260) + nv * (20 + 24), "flops": n * 3 * case["sweeps"] * 20}
    n = case["n"]
    sph = 64 * (73 + 101)  # density and force interactions of a gas particle
    if kind == "sn":
        return {"bytes": (case["steps"] + 1) * n * 250 + 120 * n, "flops": (case["steps"] + 1) * n * sph}
    # interactions of a particle in a tree walk at theta = 0.5: about 64 per doubling of the particle number
    pairs = n * n * 27 if case["gravity"] == "direct" else n * 64 * math.log2(n) * (59 if case["multipole"] else 27)
    if kind == "gravity":
        return {"bytes": n * (61 + 16), "flops": pairs}
    ng = int(round(case["gas"] * n))
    return {"bytes": case["steps"] * (n * 200 + ng * 250) + n * 70, "flops": case["steps"] * (pairs + ng * sph)}


# ------------------------------------------------------------------ exact values
# The same results in 64 bits, with direct sums and searches over all pairs.
F8 = torch.float64
PAIRS_DIRECT = 1.2e11   # pair counts beyond which a value would take too long
PAIRS_KNN = 1.5e11


def _direct64(x, m, e, rows):
    """Softened accelerations and potentials of every particle, G = 1."""
    n = x.shape[1]
    a, ph = torch.empty((3, n), device=DEV, dtype=F8), torch.empty(n, device=DEV, dtype=F8)
    e2 = e * e
    for i in range(0, n, rows):
        j = min(n, i + rows)
        r2 = e2[i:j, None] + e2[None, :]
        d = [x[k][None, :] - x[k][i:j, None] for k in range(3)]
        for k in range(3):
            r2.addcmul_(d[k], d[k])
        w = r2.rsqrt_()
        mw = w * m
        ph[i:j] = -(mw.sum(1) - mw[torch.arange(j - i, device=DEV), torch.arange(i, j, device=DEV)])
        mw *= w
        mw *= w
        for k in range(3):
            a[k, i:j] = (mw * d[k]).sum(1)
    return a, ph


def _knn64(x):
    """Indices and squared distances of the 64 nearest particles (self included), nearest first."""
    n = x.shape[1]
    idx, d2 = torch.empty((n, 64), device=DEV, dtype=torch.int64), torch.empty((n, 64), device=DEV, dtype=F8)
    rows = max(1, min(n, int(3e8 // n)))
    for i in range(0, n, rows):
        j = min(n, i + rows)
        d = torch.zeros((j - i, n), device=DEV, dtype=F8)
        for k in range(3):
            t = x[k][None, :] - x[k][i:j, None]
            d.addcmul_(t, t)
        v = torch.topk(d, 64, largest=False, sorted=True)
        idx[i:j], d2[i:j] = v.indices, v.values
    return idx, d2


def _kern(q):
    return torch.where(q <= 0.5, 1 - 6 * q ** 2 + 6 * q ** 3, torch.where(q <= 1, 2 * (1 - q) ** 3, 0.0))


def _dkern(q):
    return torch.where(q <= 0.5, -12 * q + 18 * q ** 2, torch.where(q <= 1, -6 * (1 - q) ** 2, 0.0))


def _density64(x, m, u, pressure):
    gamma = 5.0 / 3.0
    idx, d2 = _knn64(x)
    h2 = d2[:, 63]
    h = torch.sqrt(h2)
    w = m[idx] * _kern(torch.sqrt(d2) / h[:, None]) * (8.0 / math.pi) / h[:, None] ** 3
    rho = w.sum(1)
    P = (gamma - 1) * ((w * u[idx]).sum(1) if pressure else rho * u)
    return {"idx": idx, "d2": d2, "h2": h2, "h": h, "rho": rho, "P": P, "cs": torch.sqrt(gamma * P / rho)}


def _hydro64(x, v, u, m, D, pressure):
    """Accelerations, du/dt and the largest signal velocities over the symmetric neighbour sets."""
    gamma, n = 5.0 / 3.0, x.shape[1]
    rep = torch.arange(n, device=DEV)[:, None].expand(n, 64)
    own = D["idx"] != rep
    i, j = rep[own], D["idx"][own]
    one = D["d2"][own] > D["h2"][j]  # i is not among the neighbours of j: the pair counts for j too
    i, j = torch.cat([i, j[one]]), torch.cat([j, i[one]])
    d = [x[k][i] - x[k][j] for k in range(3)]
    r = torch.sqrt(d[0] ** 2 + d[1] ** 2 + d[2] ** 2)
    rinv = torch.where(r > 0, 1.0 / r, 0.0)
    h, rho, P, cs = D["h"], D["rho"], D["P"], D["cs"]
    dwi, dwj = (_dkern(r / h[k]) * (8.0 / math.pi) / h[k] ** 4 for k in (i, j))
    w = sum((v[k][i] - v[k][j]) * d[k] for k in range(3)) * rinv
    vs = cs[i] + cs[j] - 3.0 * w.clamp_max(0.0)
    visc = torch.where(w < 0, -0.5 * vs * w / (0.5 * (rho[i] + rho[j])), 0.0)
    if pressure:
        uu = (gamma - 1) ** 2 * u[i] * u[j]
        ci, cj = uu / P[i], uu / P[j]
    else:
        ci, cj = P[i] / rho[i] ** 2, P[j] / rho[j] ** 2
    bar = 0.5 * (dwi + dwj)
    f = -m[j] * (ci * dwi + cj * dwj + visc * bar) * rinv
    a = torch.zeros((3, n), device=DEV, dtype=F8)
    for k in range(3):
        a[k].index_add_(0, i, f * d[k])
    du = torch.zeros(n, device=DEV, dtype=F8).index_add_(0, i, m[j] * (ci * dwi + 0.5 * visc * bar) * w)
    vsig = (2.0 * cs).scatter_reduce(0, i, vs, "amax")
    return a, du, vsig


def _forces64(x, v, u, p, case, halo):
    """Total acceleration, potential, du/dt and the gas fields; v and u are those the SPH terms see."""
    n = x.shape[1]
    m, e, gas = p["m"].to(F8), p["eps"].to(F8), torch.nonzero(p["type"] == 1)[:, 0]
    a, pot = torch.zeros((3, n), device=DEV, dtype=F8), torch.zeros(n, device=DEV, dtype=F8)
    if case["kind"] != "sn":
        a, pot = _direct64(x, m, e, max(1, min(n, int(2e8 // n))))
    if halo:
        r = torch.sqrt((x * x).sum(0))
        s = r / ics.NFW_RS
        a = a - x * (ics.NFW_MS * (torch.log1p(s) - s / (1 + s)) / r ** 3)
    z = torch.zeros(n, device=DEV, dtype=F8)
    out = {"a": a, "pot": pot, "dudt": z, "rho": z.clone(), "h2": z.clone()}
    if gas.numel():
        xg, vg, ug = x[:, gas], v[:, gas], u[gas]
        D = _density64(xg, m[gas], ug, case["pressure"])
        ah, du, vsig = _hydro64(xg, vg, ug, m[gas], D, case["pressure"])
        out["a"] = a.index_add(1, gas, ah)
        out["dudt"] = z.index_add(0, gas, du)
        out["rho"][gas], out["h2"][gas] = D["rho"], D["h2"]
        out["dt"] = float((D["h"] / vsig).min())
    return out


def _leapfrog64(case, p):
    x = torch.stack([p["x"], p["y"], p["z"]])
    v = torch.stack([p["vx"], p["vy"], p["vz"]]).to(F8)
    u = p["u"].to(F8)
    halo, t, steps = bool(_halo(case)), 0.0, 0
    F = _forces64(x, v, u, p, case, halo)
    for _ in range(case["steps"]):
        dt = DT if case["kind"] == "step" else min(0.3 * F["dt"], ics.T_SN_END - t)
        v, u = v + 0.5 * dt * F["a"], u + 0.5 * dt * F["dudt"]
        x = x + dt * v
        F = _forces64(x, v + 0.5 * dt * F["a"], u + 0.5 * dt * F["dudt"], p, case, halo)
        v, u = v + 0.5 * dt * F["a"], u + 0.5 * dt * F["dudt"]
        t, steps = t + dt, steps + 1
    val = {"X": x[0], "Y": x[1], "Z": x[2], "VX": v[0], "VY": v[1], "VZ": v[2], "U": u, "AX": F["a"][0],
           "AY": F["a"][1], "AZ": F["a"][2], "POT": F["pot"], "DUDT": F["dudt"], "RHO": F["rho"], "H2": F["h2"]}
    return val, t, steps


def _voxelise64(case, p):
    G, d, out, at = case["grid"], SIDE / case["grid"], [], 0
    for n, c in zip(_sizes(case), _centres(case)):
        sl = slice(at, at + n)
        at += n
        x = torch.stack([p[k][sl] - (c[a] - 0.5 * SIDE) for a, k in enumerate("xyz")])
        v = torch.stack([p[k][sl].to(F8) for k in ("vx", "vy", "vz")])
        m, u = p["m"][sl].to(F8), p["u"][sl].to(F8)
        D = _density64(x, m, u, False)
        term = torch.cat([torch.stack([m, m / D["rho"], u * ics.T_PER_U * m / D["rho"]]), v * (m / D["rho"])])
        acc = torch.zeros((6, G ** 3), device=DEV, dtype=F8)
        base, reach = torch.floor(x / d).to(torch.int64), torch.ceil(D["h"] / d + 0.5).to(torch.int64)
        for r in range(1, int(reach.max()) + 1):
            who = torch.nonzero(reach == r)[:, 0]
            o = torch.arange(-r, r + 1, device=DEV)
            off = torch.stack(torch.meshgrid(o, o, o, indexing="ij")).reshape(3, 1, -1)
            step = max(1, int(2e7 // off.shape[2]))
            for q in who.split(step):
                ijk = base[:, q, None] + off
                r2 = (((ijk + 0.5) * d - x[:, q, None]) ** 2).sum(0)
                hq = D["h"][q, None]
                hit = (r2 < hq * hq) & (ijk >= 0).all(0) & (ijk < G).all(0)
                w = (_kern(torch.sqrt(r2) / hq) * (8.0 / math.pi) / hq ** 3)[hit]
                vox = ((ijk[2] * G + ijk[1]) * G + ijk[0])[hit]
                part = torch.nonzero(hit)[:, 0]
                for k in range(6):
                    acc[k].index_add_(0, vox, term[k][q][part] * w)
        den = acc[1]
        some, safe = den > 0, torch.where(den > 0, den, 1.0)
        T = torch.where(some, acc[2] / safe, 10.0)
        z = [torch.log10(acc[0].clamp_min(1e-4)) + 0.33, (torch.log10(T.clamp_min(10.0)) - 2.0) / 2.0]
        out.append(torch.stack(z + [torch.where(some, acc[k] / safe, 0.0) / 20.0 for k in (3, 4, 5)], 1))
    return torch.stack(out)


def _i64(v):
    return v - (1 << 64) if v >> 63 else v


def _mix64(x):
    """SplitMix64 of 64-bit integers held in int64 tensors."""
    def shr(a, k):
        return (a >> k) & ((1 << (64 - k)) - 1)
    z = x + _i64(0x9E3779B97F4A7C15)
    z = (z ^ shr(z, 30)) * _i64(0xBF58476D1CE4E5B9)
    z = (z ^ shr(z, 27)) * _i64(0x94D049BB133111EB)
    return z ^ shr(z, 31)


def _uniform64(sid, k):
    return ((_mix64(sid + k) >> 11) & ((1 << 53) - 1)).to(F8) * 2.0 ** -53


def _remap64(case, p, pred, seed):
    """Positions, velocities and internal energies after the Gibbs sampling."""
    G, d, at = case["grid"], SIDE / case["grid"], 0
    res = {k: [] for k in ("X", "Y", "Z", "VX", "VY", "VZ", "U")}
    for reg, (n, c) in enumerate(zip(_sizes(case), _centres(case))):
        sl = slice(at, at + n)
        at += n
        w = (10.0 ** (pred[reg, :, 0].to(F8) - 0.33)).reshape(G, G, G)  # z, y, x
        cdf = [torch.cumsum(w, 2), torch.cumsum(w, 1).permute(0, 2, 1), torch.cumsum(w, 0).permute(1, 2, 0)]
        cdf = [t.contiguous() for t in cdf]
        lo = [c[a] - 0.5 * SIDE for a in range(3)]
        vox = [torch.floor((p[k][sl] - lo[a]) / d).clamp(0, G - 1).to(torch.int64) for a, k in enumerate("xyz")]
        sid = _mix64(p["id"][sl] + seed)
        for k in range(3 * case["sweeps"]):
            a = k % 3
            line = cdf[a][vox[2] if a < 2 else vox[1], vox[1] if a == 0 else vox[0]]
            target = _uniform64(sid, k) * line[:, -1]
            vox[a] = (line <= target[:, None]).sum(1).clamp_max(G - 1)
        for a, k in enumerate("XYZ"):
            res[k].append(lo[a] + (vox[a] + _uniform64(sid, 3 * case["sweeps"] + a)) * d)
        v = pred[reg].to(F8)[(vox[2] * G + vox[1]) * G + vox[0]]
        res["U"].append(10.0 ** (2.0 * v[:, 1] + 2.0) / ics.T_PER_U)
        for a, k in enumerate(("VX", "VY", "VZ")):
            res[k].append(20.0 * v[:, 2 + a])
    return dict({k: torch.cat(t) for k, t in res.items()}, KEY=None, ORDER=None)


def _conv64(x, w, b, G):
    """3^3 convolution, zero padding, of [voxels z y x, cin] by [27, cin, cout]."""
    xp = torch.nn.functional.pad(x.reshape(-1, G, G, G, x.shape[1]), (0, 0, 1, 1, 1, 1, 1, 1))
    y = b.expand(x.shape[0], w.shape[2]).clone()
    for t in range(27):
        z0, y0, x0 = t // 9, t // 3 % 3, t % 3
        y = y + xp[:, z0:z0 + G, y0:y0 + G, x0:x0 + G].reshape(x.shape[0], -1) @ w[t]
    return y


def _unet64(case, layers, x):
    L, G = case["levels"], case["grid"]
    it = iter(layers)
    B, act, skip = x.shape[0], x.reshape(-1, 5), []
    for l in range(L):
        g = G >> l
        for _ in range(2):
            act = torch.relu(_conv64(act, *next(it), g))
        if l + 1 < L:
            skip.append(act)
            act = act.reshape(B, g // 2, 2, g // 2, 2, g // 2, 2, -1).amax((2, 4, 6)).reshape(-1, act.shape[1])
    for l in range(L - 2, -1, -1):
        g = G >> l
        w, b = next(it)
        up = torch.einsum("vc,tco->vto", act, w) + b
        up = up.reshape(B, g // 2, g // 2, g // 2, 2, 2, 2, -1).permute(0, 1, 4, 2, 5, 3, 6, 7).reshape(-1, w.shape[2])
        act = torch.cat([skip[l], up], 1)
        for _ in range(2):
            act = torch.relu(_conv64(act, *next(it), g))
    w, b = next(it)
    return (act @ w[0] + b).reshape(x.shape[:4] + (5,))


def _unet_exact(case, seed):
    _, flat = _net(case, seed)
    x, t = _grids(case, seed)
    flat = torch.from_numpy(flat).to(DEV, F8).requires_grad_(case["kind"] == "train")
    layers, at = [], 0
    for k, ci, co, _ in _net_shape(case):
        nt = {"conv": 27, "up": 8, "head": 1}[k]
        layers.append((flat[at:at + nt * ci * co].reshape(nt, ci, co), flat[at + nt * ci * co:at + nt * ci * co + co]))
        at += nt * ci * co + co
    if case["kind"] == "forward":
        return torch.cat([_unet64(case, layers, x[b:b + 1].to(F8)) for b in range(case["batch"])])
    loss = ((_unet64(case, layers, x.to(F8)) - t.to(F8)) ** 2).mean()
    loss.backward()
    g = flat.grad
    # Adam's first step: both moments' bias corrections cancel
    return {"loss": float(loss.detach()), "grads": g, "params": flat.detach() - 1e-3 * g / (g.abs() + 1e-8)}


def exact(case, seed):
    kind = case["kind"]
    if kind in ("forward", "train"):
        return _unet_exact(case, seed)
    if kind == "remap":
        return _remap64(case, _particles(case, seed), _prediction(case, seed), int(seed))
    if kind == "voxelise":
        if sum(float(n) ** 2 for n in _sizes(case)) > PAIRS_KNN:
            return None
        return _voxelise64(case, _particles(case, seed))
    n = float(case["n"])
    if kind == "sn":
        if (case["steps"] + 1) * n * n > PAIRS_KNN:
            return None
        val, t, steps = _leapfrog64(case, _particles(case, seed))
        return dict({k: val[k] for k in SN_FIELDS}, steps=None, t=t)
    evaluations = case["steps"] + 1 if kind == "step" else 1
    if evaluations * n * n > PAIRS_DIRECT:
        return None
    p = _particles(case, seed)
    if kind == "gravity":
        x = torch.stack([p["x"], p["y"], p["z"]])
        a, pot = _direct64(x, p["m"].to(F8), p["eps"].to(F8), max(1, min(int(n), int(2e8 // n))))
        return {"AX": a[0], "AY": a[1], "AZ": a[2], "POT": pot}
    val = _leapfrog64(case, p)[0]
    return {k: val[k] for k in (STEP_FIELDS if case["gas"] else STAR_FIELDS)}
