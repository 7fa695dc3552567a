"""Calls that fail part-way: what they leave behind.

Device allocations are made to fail on the host (gnb_test_fail_alloc), one
after the other, and a sort is told that a wait ran out
(gnb_test_sort_give_up); nothing here makes a kernel fault or hang."""
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


FIELDS = ("X", "Y", "Z", "AX", "AY", "AZ", "POT", "DUDT", "RHO", "H2")


def _calls(G, c, net, p, cen, rep):
    return [
        lambda: c.set_particles(p),
        lambda: c.compute_forces(G.GNB_GRAV_DIRECT),
        lambda: c.compute_forces(G.GNB_GRAV_TREE),
        lambda: c.voxelise([cen], grid=12),
        lambda: c.sn_async_submit(net, [cen], seed=3, sweeps=1),
        lambda: c.sn_async_apply(),
        lambda: c.replace_region(rep),
        lambda: c.compute_forces(G.GNB_GRAV_TREE),
    ]


def test_calls_after_a_failed_allocation(G):
    """Whichever allocation of a context fails, the call that made it returns
    GNB_ENOMEM and the same call works when it is repeated: no array is used
    whose replacement was not allocated, and the results are those of a
    context without a failure."""
    from paper_2510_23330_gb300 import surrogate
    n, cen, big = 2000, (0.0, 0.0, 0.0), 1 << 40
    p = ics.sn_region(n, seed=2, grid=16)
    rng = np.random.default_rng(0)
    pick = rng.permutation(n)[:50]
    rep = {k: p[k][pick].copy() for k in ("id", "x", "y", "z", "vx", "vy", "vz", "u")}
    for k in "xyz":
        rep[k] += rng.uniform(-1.0, 1.0, 50)
    net = G.UNet(5, 5, 16, 2, 8)
    net.set_params(surrogate.he_init(5, 5, 16, 2, seed=1))

    def run(after):
        c = G.Context()
        G.gnb_test_fail_alloc(c.h, after)
        failed = 0
        for call in _calls(G, c, net, p, cen, rep):
            try:
                call()
            except G.GalnbError as e:
                assert e.code == G.GNB_ENOMEM and failed == 0
                failed += 1
                call()
        out = {k: c.get(k).astype(np.float64) for k in FIELDS}
        if after < big:
            # from arrays of this size to larger ones: everything is replaced once more
            assert failed == 1
            c.set_particles({k: np.concatenate([v, v]) for k, v in p.items()})
            c.compute_forces(G.GNB_GRAV_TREE)
        left = G.gnb_test_fail_alloc(c.h, -1)
        c.close()
        return out, left

    ref, left = run(big)
    for after in range(big - left):
        got, _ = run(after)
        for k in FIELDS:
            # (the symmetric SPH sums have no fixed order)
            assert np.max(np.abs(got[k] - ref[k])) <= 1e-4 * np.max(np.abs(ref[k])), (after, k)


@pytest.mark.parametrize("n_gas", [0, 500])
def test_list_pool_that_cannot_grow(G, n_gas):
    """A nearly direct walk of small groups over single-particle leaves outgrows
    the first interaction-list pool; when the larger one cannot be allocated
    the accelerations were never evaluated and are not handed out, and the next
    call finds memory again."""
    p = ics.plummer(6000, seed=2, n_gas=n_gas)
    names = ("AGRAV_X", "AGRAV_Y", "AGRAV_Z", "POT", "AX")
    c, d = G.Context(theta=0.03, n_leaf=1, n_group=8), G.Context(theta=0.03, n_leaf=1, n_group=8)
    for q in (c, d):
        q.set_particles(p)
        q.compute_sph_density()  # every other array of the calls below
    call = {0: "compute_gravity", 500: "compute_forces"}[n_gas]
    G.gnb_test_fail_alloc(c.h, 6)  # the pool's six arrays, not the larger pool
    with pytest.raises(G.GalnbError) as e:
        getattr(c, call)(G.GNB_GRAV_TREE)
    assert e.value.code == G.GNB_ENOMEM and G.gnb_test_fail_alloc(c.h, -1) == -1
    for k in names:
        with pytest.raises(G.GalnbError) as e:
            c.get(k)
        assert e.value.code == G.GNB_ESTATE
    with pytest.raises(G.GalnbError):
        c.diagnostics()
    if n_gas:
        c.compute_sph_force()  # of the density that was there; not a force to step with
        with pytest.raises(G.GalnbError):
            c.get("POT")
    for q in (c, d):
        getattr(q, call)(G.GNB_GRAV_TREE)
    for k in names:
        assert np.allclose(c.get(k), d.get(k), rtol=1e-5, atol=1e-6)
    d.compute_gravity(G.GNB_GRAV_DIRECT)
    assert np.median(np.abs(c.get("AGRAV_X") / d.get("AGRAV_X") - 1.0)) < 1e-4


def test_search_that_fails_leaves_the_supports(G, tmp_path):
    """Three hundred gas particles at one point cannot be ranked: the
    kernel-size search fails for them, after it has found the supports of the
    others.  The supports of the state stay those it came with, and the density
    of the failed call is not handed out."""
    p = ics.sn_region(3000, seed=4, grid=16)
    for k in "xyz":
        p[k][:300] = p[k][0]
    n = p["x"].size
    rng = np.random.default_rng(1)
    p["h2"] = rng.uniform(1.0, 2.0, n)
    for k in ("ax", "ay", "az", "dudt"):
        p[k] = np.zeros(n, np.float32)
    c = G.Context()
    c.set_state(p, G.GNB_GRAV_NONE)
    for call in (c.compute_sph_density, lambda: c.compute_forces(G.GNB_GRAV_NONE)):
        with pytest.raises(G.GalnbError) as e:
            call()
        assert e.value.code == G.GNB_ECAPACITY
        for k in ("RHO", "H2", "NBR"):
            with pytest.raises(G.GalnbError):
                c.get(k)
        path = str(tmp_path / "state")
        c.save(path)
        # after the header: id, type, 3 positions, 6 floats, then h2 and 12 floats
        raw = open(path, "rb").read()
        at = len(raw) - n * (8 + 12 * 4)
        assert np.array_equal(np.frombuffer(raw, np.float64, n, at), p["h2"])


def test_hydro_calls_on_a_loaded_state(G, tmp_path):
    """A saved state holds no neighbour lists and no signal velocities: the
    calls that need them, on the state just loaded, give what they give in the
    context that saved it."""
    p, path = ics.plummer(4000, seed=6, n_gas=1500), str(tmp_path / "state")
    a = G.Context()
    a.set_particles(p)
    a.compute_gravity(G.GNB_GRAV_TREE)
    a.compute_sph_density()
    a.save(path)
    a.compute_sph_force()
    dt = a.cfl_timestep()
    names = ("AX", "AY", "AZ", "DUDT", "RHO", "H2")
    ref = {k: a.get(k) for k in names}

    b = G.Context()
    b.load(path)
    b.compute_sph_force()
    for k in names:  # (sums of the symmetric force have no fixed order)
        assert np.max(np.abs(b.get(k) - ref[k])) <= 1e-5 * np.max(np.abs(ref[k])), k
    assert abs(b.cfl_timestep() - dt) <= 1e-5 * dt

    a.save(path)
    b = G.Context()
    b.load(path)
    assert np.array_equal(b.get("AX"), ref["AX"])
    assert abs(b.cfl_timestep() - dt) <= 1e-5 * dt
    b = G.Context()
    b.load(path)
    for c in (a, b):
        assert c.integrate_cfl(1.5 * dt, mode=G.GNB_GRAV_TREE)[1] == 2
    for k in ("X", "VX", "U"):
        assert np.allclose(a.get(k), b.get(k), rtol=1e-4, atol=1e-6)

    # results that came with a state do not follow its particles into the sorted order
    b = G.Context()
    b.load(path)
    b.compute_sph_density()
    with pytest.raises(G.GalnbError):
        b.get("AX")


@pytest.mark.parametrize("last", [2, 4, 7])
def test_sort_that_gave_up(G, orc, last):
    """After a pass whose wait ran out the later passes leave their arrays
    alone (places that were never written have other digits than were
    counted); the call reports it and the next one sorts."""
    p = ics.plummer(5000, seed=last, n_gas=0)
    c = G.Context()
    c.set_particles(p)
    assert G.gnb_test_sort_give_up(c.h, last) == G.GNB_OK
    with pytest.raises(G.GalnbError) as e:
        c.build_tree()
    assert e.value.code == G.GNB_ETIMEOUT
    for k in ("KEY", "NODES"):
        with pytest.raises(G.GalnbError):
            c.get(k)
    c.build_tree()
    key, _, _, _ = orc.morton(p)
    assert np.array_equal(c.get("KEY"), key.astype(np.int64))
    assert np.array_equal(c.get("ORDER"), orc.sort_order(key))


def test_upload_of_arrays_that_are_not_all_there(G):
    """Device arrays are read in place only where the whole of each lies in one
    allocation: pinned and managed memory is taken as before, an array of half
    the length is refused by the copy it then goes through."""
    import ctypes as C
    import torch
    p = ics.plummer(1 << 15, seed=1, n_gas=0)
    n = p["x"].size
    dev = {k: torch.from_numpy(np.ascontiguousarray(p[k], dtype=t)).cuda() for k, t in G.Context._DT.items()}
    managed, half = C.c_void_p(), C.c_void_p()
    L = G.lib()
    assert L.cudaMallocManaged(C.byref(managed), C.c_size_t(8 * n), 1) == 0
    assert L.cudaMalloc(C.byref(half), C.c_size_t(4 * n)) == 0
    C.memmove(managed, p["x"].ctypes.data, 8 * n)
    pinned = torch.from_numpy(p["x"].copy()).pin_memory()
    torch.cuda.synchronize()
    for x, ok in ((dev["x"].data_ptr(), True), (pinned.data_ptr(), True), (managed.value, True), (half.value, False)):
        c = G.Context()
        c.n = n
        rc = G.gnb_set_particles(c.h, n, *[x if k == "x" else dev[k].data_ptr() for k in dev], 1)
        assert rc == (G.GNB_OK if ok else G.GNB_ECUDA)
        if not ok:  # and the refused call leaves nothing for the next
            c.set_particles(p)
        assert np.array_equal(c.get("X"), p["x"])
        c.close()
    assert L.cudaFree(managed) == 0 and L.cudaFree(half) == 0


def test_particle_inside_a_thin_shell(G, orc):
    """A particle that sees its 64th neighbour among equal distances: 60 in a
    shell a millionth thick are ranked, 200 are more than the uncertain entries
    that can be (they fail at once: the band of the 64th reaches past the list)."""
    rng = np.random.default_rng(3)
    for m, ok in ((60, True), (200, False)):
        p = ics.uniform_random(4000, seed=9)
        x = np.stack([p[k] for k in "xyz"], axis=1)
        at = x.mean(0)
        far = np.argsort(((x - at) ** 2).sum(1))[::-1]
        hole = 0.5 * np.sqrt(((x - at) ** 2).sum(1)).max()
        d = x - at
        r = np.sqrt((d**2).sum(1))
        x = at + d * np.maximum(1.0, hole / np.maximum(r, 1e-12))[:, None] * rng.uniform(1.0, 1.2, (x.shape[0], 1))
        x[far[0]] = at
        v = rng.normal(size=(m, 3))
        x[far[1 : m + 1]] = at + 0.4 * hole * (1.0 + 5e-7 * rng.uniform(-1.0, 1.0, (m, 1))) * v / np.sqrt((v**2).sum(1))[:, None]
        for k, a in zip("xyz", range(3)):
            p[k] = np.ascontiguousarray(x[:, a])
        c = G.Context()
        c.set_particles(p)
        if ok:
            c.compute_sph_density()
            d2 = np.sort(((x - at) ** 2).sum(1))
            assert abs(c.get("H2")[far[0]] - d2[63]) < 1e-12 * d2[63]
        else:
            with pytest.raises(G.GalnbError) as e:
                c.compute_sph_density()
            assert e.value.code == G.GNB_ECAPACITY


@pytest.mark.parametrize("n", [100, 250000])
def test_scratch_of_the_sort_comes_with_the_particles(G, n):
    """The first tree of a context allocates the tree's twelve arrays and
    nothing else, also for fewer particles than the context has held, and the
    sort still orders them."""
    big = 1 << 40
    p = ics.uniform_random(n, seed=n, gas_frac=0.0)
    c = G.Context()
    c.set_particles(ics.uniform_random(n + 1, seed=1, gas_frac=0.0))
    c.set_particles(p)
    G.gnb_test_fail_alloc(c.h, big)
    c.build_tree()
    assert big - G.gnb_test_fail_alloc(c.h, -1) == 12
    key = c.get("KEY")
    assert np.array_equal(c.get("ORDER"), np.lexsort((np.arange(n), key)))


@pytest.mark.parametrize("change", ["kernels", "buffers"])
def test_captured_batch_follows_the_network(G, change):
    """The graph of a surrogate batch holds the network's buffers and kernels:
    after another choice of kernels, or a larger batch that moved the buffers,
    the next call captures again instead of replaying what is no longer there."""
    import torch
    from paper_2510_23330_gb300 import surrogate
    stream = torch.cuda.Stream()
    p, cen = ics.sn_region(3000, seed=5, grid=16), [(0.0, 0.0, 0.0)]
    with torch.cuda.stream(stream):
        net = G.UNet(5, 5, 16, 2, 8, stream=stream.cuda_stream)
        net.set_params(surrogate.he_init(5, 5, 16, 2, seed=1))
        c = G.Context(stream=stream.cuda_stream)
        out, launches = [], []
        for step in range(3):
            if step == 2 and change == "kernels":
                net.set_conv_impl(G.GNB_CONV_MMA_SYNC)
            elif step == 2:
                net.forward(np.zeros((40, 8, 8, 8, 5), np.float32))
            c.set_particles(p)
            c.compute_sph_density()
            before = c.phase_times()[2]
            c.sn_surrogate_batch(net, cen, seed=3, sweeps=0, use_graph=True)
            launches.append(c.phase_times()[2] - before)
            out.append({k: c.get(k).astype(np.float64) for k in ("X", "U")})
        stream.synchronize()
    assert launches[0] > 10 and launches[1] == 0 and launches[2] > 10
    for o in out[1:]:
        assert np.array_equal(o["X"], out[0]["X"])  # no sweeps: positions do not depend on the prediction
        assert np.all(np.abs(np.log10(o["U"] / out[0]["U"])) < 0.3)
