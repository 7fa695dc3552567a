"""GPU paths chosen by size, at the sizes where the choice or a tile ends."""
import numpy as np
import pytest

from paper_2510_23330_gb300 import ics

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def G():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2510_23330_gb300 import galnb
    return galnb


# tree build: one round of 256 slots per tile up to 2^20 slots, two beyond
@pytest.mark.parametrize("n", [255, 256, 257, (1 << 20) + 1])
def test_tree_topology_at_tile_edges(G, orc, n):
    p = ics.plummer(n, seed=n, n_gas=0)
    c = G.Context(n_leaf=16, n_group=64)
    c.set_particles(p)
    c.build_tree()
    key, _, _, _ = orc.morton(p)
    tree = orc.octree(key[orc.sort_order(key)], 16)
    ref = np.stack([tree["level"], tree["prefix"].astype(np.int64), tree["first"], tree["count"]], axis=1)
    assert np.array_equal(c.get("NODES"), ref)
    links = c.get("NODE_LINKS").reshape(-1, 3)
    assert np.array_equal(links[:, 0], tree["child"]) and np.array_equal(links[:, 1], tree["nchild"])
    assert np.array_equal(np.sort(c.get("GROUPS")), np.sort(orc.groups(tree, 64)))


def _clump(seed):
    """A dense ball inside a wide one: runs whose candidates overflow, and outer
    particles that see the ball as a thin shell."""
    rng = np.random.default_rng(seed)
    d = rng.normal(size=(1400, 3))
    d /= np.linalg.norm(d, axis=1, keepdims=True)
    r = np.where(np.arange(1400) < 1200, 1e-3, 3.0) * rng.uniform(0.0, 1.0, 1400) ** (1.0 / 3.0)
    p = ics.uniform_random(1400, seed=seed)
    x = d * r[:, None] + 0.3
    return dict(p, x=x[:, 0].copy(), y=x[:, 1].copy(), z=x[:, 2].copy())


# kernel-size search: the smallest sets, runs of 1 | 2 and 2 | 4 particles (4
# and 12 gas particles per resident warp of 152 SMs x 24), and a clump; then
# the same particles spread out, so that every support outgrows its search
# radius
@pytest.mark.parametrize("case", [64, 66, 14592, 14593, 43777, "clump"])
def test_kernel_sizes_exact_twice(G, orc, case):
    p = _clump(5) if case == "clump" else ics.uniform_random(case, seed=case)
    n = p["x"].size
    rng = np.random.default_rng(1)
    sample = np.arange(n) if n <= 2000 else np.sort(rng.choice(n, 600, replace=False))
    c = G.Context()
    c.set_particles(p)
    for k in range(2):
        if k:
            s = 1.0 + 0.7 * rng.uniform(0.9, 1.1)
            p = dict(p, x=s * p["x"], y=s * p["y"], z=1.1 * s * p["z"])
            c.replace_region({q: p[q] for q in ("id", "x", "y", "z", "vx", "vy", "vz", "u")})
        c.compute_sph_density()
        nbr, h2 = orc.knn({q: np.asarray(p[q], np.float64) for q in ("x", "y", "z", "m", "u")}, 64, sample=sample)
        assert np.array_equal(c.get("NBR")[sample], np.sort(nbr, axis=1))
        assert np.array_equal(c.get("H2")[sample], h2)


# hydro force: 16 and 8 lanes per particle below 150,000 gas particles, 8 and 4
# from there.  Equal and opposite pairs: any pair lost, doubled or one-sided
# shows in the totals of momentum and energy.
@pytest.mark.parametrize("n", [64, 67, 149999, 150001])
@pytest.mark.parametrize("variant", [0, 1])
def test_hydro_force_conserves(G, n, variant):
    p = ics.uniform_random(n, seed=n)
    c = G.Context(sph_variant=variant)
    c.set_particles(p)
    c.compute_sph_density()
    c.compute_sph_force()
    m, du = p["m"].astype(np.float64), c.get("DUDT").astype(np.float64)
    a = np.stack([c.get(k) for k in ("AX", "AY", "AZ")]).astype(np.float64)
    v = np.stack([p[k] for k in ("vx", "vy", "vz")]).astype(np.float64)
    force = np.sum(m * np.linalg.norm(a, axis=0))
    # FP32 sums of ~70 terms per particle, errors independent between particles
    assert np.linalg.norm((m * a).sum(1)) < 1e-5 * force
    power = np.sum(m * (np.abs(du) + np.linalg.norm(a, axis=0) * np.linalg.norm(v, axis=0)))
    assert abs(np.sum(m * ((a * v).sum(0) + du))) < 1e-5 * power
    nb = c.get("NBR")
    pairs = set()
    if n < 1000:  # the symmetric lists hold 63 own entries and the one-sided pairs once more
        pairs = {(i, j) for i in range(n) for j in nb[i] if i != j}
        assert c.stats()["NSYM"] == 63 * n + sum((j, i) not in pairs for i, j in pairs)


# radix sort: one tile, tile edges, 4 | 8 | 16 pairs per thread of a tile, and
# a run of equal keys longer than the tie pass takes (whole-key sort)
@pytest.mark.parametrize("n", [1, 1023, 1024, 1025, 200001, 500001, "ties"])
def test_sort_order(G, orc, n):
    p = ics.plummer(9000 if n == "ties" else max(n, 4), seed=3, n_gas=0)
    if n == "ties":
        for k in ("x", "y", "z"):
            p[k][1000:6000] = p[k][1000]
    elif n < 4:
        p = ics.subset(p, range(n))
    c = G.Context()
    c.set_particles(p)
    for k in range(2):  # from the caller's order, then from the sorted one
        c.build_tree()
        key = orc.morton(p)[0]
        assert np.array_equal(c.get("KEY"), key)
        assert np.array_equal(c.get("ORDER"), np.lexsort((np.arange(key.size), key)))
        assert np.array_equal(c.get("X"), p["x"]) and np.array_equal(c.get("VZ"), p["vz"])
        rng = np.random.default_rng(k)
        p = dict(p, x=p["x"] + 1e-3 * rng.normal(size=key.size))
        c.replace_region({q: p[q] for q in ("id", "x", "y", "z", "vx", "vy", "vz", "u")})


# direct gravity: one and several parts of the sources, one, two and four
# particles per thread, a group above 512, the three softening forms
@pytest.mark.parametrize("n,n_group", [(513, 8), (1023, 64), (1025, 600), (2500, 2500)])
@pytest.mark.parametrize("eps", ["uniform", "mixed", "zero"])
def test_direct_gravity_forms(G, orc, n, n_group, eps):
    p = ics.plummer(n, seed=n, n_gas=0)
    rng = np.random.default_rng(n)
    if eps != "uniform":
        p["eps"] = (0.02 * rng.uniform(0.2, 1.0, n)).astype(np.float32)
    if eps == "zero":
        p["eps"][::3] = 0.0
    c = G.Context(n_group=n_group)
    c.set_particles(p)
    c.compute_gravity(G.GNB_GRAV_DIRECT)
    ref = orc.direct_gravity(p)
    d = np.sqrt(sum((c.get("AGRAV_" + k) - ref["a" + k.lower()]) ** 2 for k in "XYZ"))
    assert np.max(d / ref["asum"]) < 1e-5


# upload: the gas ranks and the copy from device arrays around block chunks, a
# mixed set, and device arrays that start at odd addresses; export of more
# fields than one launch takes
@pytest.mark.parametrize("n", [65, 256 * 912 - 1, 256 * 912 + 1])
def test_upload_and_export(G, n):
    import torch
    p = ics.uniform_random(n, seed=n)
    p["type"] = (np.random.default_rng(n).uniform(size=n) < 0.7).astype(np.uint8) if n > 100 else p["type"]
    size = {k: v.dtype.itemsize for k, v in p.items()}
    dev = {k: torch.from_numpy(v).cuda() for k, v in p.items()}
    raw = {k: torch.empty(n * size[k] + 1, dtype=torch.uint8, device="cuda") for k in p}  # off by one byte
    for k in p:
        raw[k][1:] = dev[k].view(torch.uint8).reshape(-1)
    keys = ("id", "type", "x", "y", "z", "vx", "vy", "vz", "m", "eps", "u")
    out = []
    for how in ("host", "device", "odd"):
        c = G.Context()
        if how == "odd":
            torch.cuda.synchronize()
            assert G.gnb_set_particles(c.h, n, *[raw[k].data_ptr() + 1 for k in keys], 1) == 0
            c.n, c.n_gas = n, int(p["type"].sum())
        else:
            c.set_particles(p if how == "host" else dev)
        assert c.stats()["NGAS"] == int(p["type"].sum())
        c.build_tree()
        f = {k: torch.empty(n, device="cuda", dtype=torch.float64 if k in "XYZ" else torch.int64 if k == "ID" else
                            torch.float32) for k in ("X", "Y", "Z", "VX", "VY", "VZ", "U", "ID")}
        c.get_fields(f)
        fids, reps = [G.F["VX"], G.F["X"]] * 20, [torch.empty(n, device="cuda", dtype=torch.float64) for _ in range(40)]
        import ctypes as C
        assert G.gnb_get_fields(c.h, 40, (C.c_int * 40)(*fids), (C.c_void_p * 40)(*[r.data_ptr() for r in reps]),
                                (C.c_int64 * 40)(*[n] * 40), 1) == 0
        assert all(torch.equal(r, f["X"]) for r in reps[1::2])
        assert all(torch.equal(r.view(torch.float32)[:n], f["VX"]) for r in reps[0::2])
        c.compute_sph_density()
        out.append({k: v.cpu().numpy() for k, v in f.items()} | {"NBR": c.get("NBR"), "H2": c.get("H2")})
    for k in ("X", "Y", "Z", "VX", "VY", "VZ", "ID"):
        assert np.array_equal(out[0][k], p[k.lower()])
    assert np.array_equal(out[0]["U"], np.where(p["type"] == 1, p["u"], 0).astype(np.float32))
    for k in out[0]:
        assert np.array_equal(out[0][k], out[1][k]) and np.array_equal(out[0][k], out[2][k])


# a nearly direct walk fills the interaction-list pool: grown and repeated after
# the evaluation, before the forces are used
@pytest.mark.parametrize("n_gas", [0, 500])
def test_list_pool_grows(G, n_gas):
    p = ics.plummer(12000, seed=2, n_gas=n_gas)
    got = {}
    for theta in (0.03, 0.5):
        c = G.Context(theta=theta, n_group=64)
        c.set_particles(p)
        c.step_kdk(1e-3, 1, G.GNB_GRAV_TREE)
        got[theta] = [c.get(k).astype(np.float64) for k in ("AGRAV_X", "AGRAV_Y", "AGRAV_Z", "VX", "X")]
        if theta < 0.1:
            assert c.stats()["NPP"] + c.stats()["NPC"] > 256 * 64 * (2 * c.stats()["NODES"] + 1774)
    d = G.Context(n_group=64)
    d.set_particles(p)
    d.step_kdk(1e-3, 1, G.GNB_GRAV_DIRECT)
    ref = [d.get(k).astype(np.float64) for k in ("AGRAV_X", "AGRAV_Y", "AGRAV_Z", "VX", "X")]
    scale = np.sqrt(sum(r ** 2 for r in ref[:3]))
    err = {t: np.sqrt(sum((a - r) ** 2 for a, r in zip(g[:3], ref))) / scale for t, g in got.items()}
    assert np.median(err[0.03]) < 1e-5 < np.median(err[0.5])
    assert np.max(np.abs(got[0.03][3] - ref[3])) < 1e-6 and np.max(np.abs(got[0.03][4] - ref[4])) < 1e-8


def _bf16(a):
    import torch
    return torch.from_numpy(np.ascontiguousarray(a, np.float32)).bfloat16().float().numpy()


# the head for every output count and width, ragged blocks and several batch
# entries: forward from the stored last activation, weight and bias gradient
# from the output gradient (BF16 operands, FP32 sums of G^3 B terms)
@pytest.mark.parametrize("base,cout", [(16, 1), (32, 2), (16, 3), (32, 4), (16, 5), (32, 6), (16, 7), (32, 8)])
def test_unet_head_forward_and_gradient(G, base, cout):
    from paper_2510_23330_gb300 import surrogate
    grid, B, rng = 20, 3, np.random.default_rng(base + cout)
    net = G.UNet(3, cout, base, 2, grid)
    w = surrogate.he_init(3, cout, base, 2, seed=cout)
    nh = base * cout + cout
    w[-cout:] = rng.normal(size=cout)
    net.set_params(w)
    x = rng.normal(size=(B, grid, grid, grid, 3)).astype(np.float32)
    t = rng.normal(size=(B, grid, grid, grid, cout)).astype(np.float32)
    y = net.forward(x)
    act = net.get_activation(8, B, grid, base).astype(np.float64)  # dec 0 b
    ref = act @ _bf16(w[-nh:-cout]).astype(np.float64).reshape(base, cout) + w[-cout:]
    assert np.max(np.abs(y - ref)) < 1e-5 * np.max(np.abs(ref))
    net.train_step(x, t, 0.0)
    g = net.get_grads()[-nh:].astype(np.float64)
    dy = _bf16(2.0 * (y - t) / y.size).astype(np.float64)
    dw = np.einsum("bzyxc,bzyxn->cn", act, dy)
    assert np.linalg.norm(g[:-cout].reshape(base, cout) - dw) < 1e-5 * np.linalg.norm(dw)
    assert np.max(np.abs(g[-cout:] - dy.sum((0, 1, 2, 3)))) < 1e-5 * np.abs(dy).sum((0, 1, 2, 3)).max()


# weight gradients of the 3^3 layers: a last voxel chunk of fewer than 64, one
# stage only, two inputs, against the mma.sync kernel on the same forward state
@pytest.mark.parametrize("grid,B", [(8, 1), (12, 3)])
def test_unet_weight_gradients_two_kernels(G, grid, B):
    from paper_2510_23330_gb300 import surrogate
    rng = np.random.default_rng(grid)
    x = rng.normal(size=(B, grid, grid, grid, 5)).astype(np.float32)
    t = rng.normal(size=x.shape).astype(np.float32)
    out = []
    for impl in (G.GNB_CONV_AUTO, G.GNB_CONV_MMA_SYNC):
        net = G.UNet(5, 5, 16, 3, grid)
        net.set_params(surrogate.he_init(5, 5, 16, 3, seed=1))
        net.set_conv_impl(impl)
        net.train_step(x, t, 0.0)
        out.append(net.get_grads().astype(np.float64))
    # both round activations to BF16; a different order of FP32 sums flips some
    assert np.linalg.norm(out[0] - out[1]) < 5e-2 * np.linalg.norm(out[1])


# the tensor-core forward with partial tiles in x, y and z, one to three levels of
# each width, and batches on both sides of the plan rule's and of the head's
# lines: every plan sums in one order, so a region's output has the same bits
# alone and in a batch; against the mma.sync kernel a sum in another order moves
# a BF16 activation by at most one place (2^-8 of it), so a tenth of the rms is
# far above what a few layers make of it and far below a wrong tap or plane
@pytest.mark.parametrize("grid,base,levels,B", [(64, 16, 4, 4), (40, 32, 3, 5), (24, 32, 4, 3), (20, 16, 3, 2)])
def test_unet_forward_plans(G, grid, base, levels, B):
    from paper_2510_23330_gb300 import surrogate
    rng = np.random.default_rng(grid + base)
    net = G.UNet(5, 5, base, levels, grid)
    net.set_params(surrogate.he_init(5, 5, base, levels, seed=2))
    x = rng.normal(size=(B, grid, grid, grid, 5)).astype(np.float32)
    y = net.forward(x)
    for b in range(B):
        assert np.array_equal(net.forward(x[b : b + 1])[0], y[b])
    net.set_conv_impl(G.GNB_CONV_MMA_SYNC)
    ref = net.forward(x[:1])[0].astype(np.float64)
    assert np.max(np.abs(y[0] - ref)) < 0.1 * np.sqrt(np.mean(ref**2))


# remap: lines with empty voxels (weight 0), weights over many decades and grids
# of each search form, against the oracle's voxel choices
@pytest.mark.parametrize("grid", [32, 64, 24])
def test_remap_extreme_weights(G, orc, grid):
    from oracle import surrogate as S
    n, side, cen, sweeps = 4000, 60.0, (3.0, 1.0, -2.0), 6
    rng = np.random.default_rng(grid)
    p = ics.sn_region(n, seed=grid, grid=16)
    for k, v in zip("xyz", cen):
        p[k] = p[k] + v
    pred = rng.normal(size=(1, grid, grid, grid, 5)).astype(np.float32)
    pred[..., 0] = rng.uniform(-25.0, 20.0, pred.shape[:-1])
    pred[..., 0][rng.uniform(size=pred.shape[:-1]) < 0.3] = -400.0
    pred[..., 0][:, : grid // 4] = 0.0
    c = G.Context()
    c.set_particles(p)
    c.remap_regions([cen], pred, side=side, seed=77, sweeps=sweeps)
    pos = np.stack([p[k] for k in "xyz"], axis=1)
    _, rp, _, _ = S.remap(pred[0].reshape(-1, 5).astype(np.float64), p["id"], pos, cen, side, grid, seed=77, sweeps=sweeps)
    got = np.stack([c.get(k) for k in "XYZ"], axis=1)
    assert np.max(np.abs(got - rp)) < 1e-12 * side


def _splitmix64(x):
    x = x + np.uint64(0x9E3779B97F4A7C15)
    x = (x ^ (x >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
    x = (x ^ (x >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
    return x ^ (x >> np.uint64(31))


# remap: draws below 2^-16 on lines whose weights add up to about 2^-89.5, just
# inside the range decided in FP32, and whose first weight is the draw's share of
# the total but for 1e-4: U times the total is a normal FP32 number only if no
# factor on the way is smaller than either
@pytest.mark.parametrize("grid", [64, 24])
def test_remap_small_draws_on_small_totals(G, orc, grid):
    from oracle import surrogate as S
    seed, n, side = 5, 200, 60.0
    rng = np.random.default_rng(grid)
    ids = np.arange(1 << 24, dtype=np.uint64)
    m = _splitmix64(_splitmix64(ids + np.uint64(seed))) >> np.uint64(11)  # 53-bit draw 0 of each ID
    ids = ids[m < (1 << 37)][:n].astype(np.int64)
    U = np.array([S.uniform(seed, int(i), 0) for i in ids])
    assert ids.size == n and np.all(U < 2.0**-16)
    line = rng.permutation(grid * grid)[:n]  # (z, y) of the particle's x line
    T = 2.0**-90 * rng.uniform(1.05, 2.0, n)
    w = np.full((grid * grid, grid), 2.0**-89.5 / (grid - 1))
    w[line, 1:] = (T / (grid - 1))[:, None]
    w[line, 0] = U * T * (1.0 + rng.choice([-1e-4, 1e-4], n))
    pred = np.zeros((1, grid, grid, grid, 5), np.float32)
    pred[..., 0] = np.log10(w).reshape(1, grid, grid, grid) + 0.33
    p = ics.sn_region(n, seed=1, grid=16)
    p["id"] = ids
    d = side / grid
    pos = np.stack([np.full(n, 5), line % grid, line // grid], axis=1) * d + 0.5 * d - 0.5 * side
    for a, k in enumerate("xyz"):
        p[k] = np.ascontiguousarray(pos[:, a])
    c = G.Context()
    c.set_particles(p)
    c.remap_regions([(0.0, 0.0, 0.0)], pred, side=side, seed=seed, sweeps=1)
    _, rp, _, _ = S.remap(pred[0].reshape(-1, 5).astype(np.float64), ids, pos, (0.0, 0.0, 0.0), side, grid, seed=seed,
                          sweeps=1)
    got = np.stack([c.get(k) for k in "XYZ"], axis=1)
    assert np.max(np.abs(got - rp)) < 1e-12 * side
