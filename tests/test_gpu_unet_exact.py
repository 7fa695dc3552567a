"""The U-Net's kernels where every sum is exact.

Networks with a few weights of +-1 per output, small whole biases and inputs,
and targets one away from the prediction: activations and activation gradients
are whole multiples of one unit small enough for BF16 (the oracle's BF16 and
FP64 results are the same numbers), and no partial sum of a weight or bias
gradient needs more than 24 bits.  FP32 accumulation in any order then gives
the oracle's numbers exactly, so a wrong tap, plane, channel group, voxel chunk
or stage of any layer is a difference, however few terms it concerns."""
import numpy as np
import pytest

from oracle import unet as U

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def G():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2510_23330_gb300 import galnb
    return galnb


CIN, COUT = 5, 4


def _params(seed, base, levels):
    rng = np.random.default_rng(seed)
    p = U.init_params(seed, CIN, COUT, base, levels)
    for k, v in p.items():
        w = np.zeros_like(v)
        if k.endswith(".b"):
            w[:] = rng.integers(0, 2, v.shape)
        else:
            T, ci, co = v.shape
            n = 4 if k == "head.w" else 2
            for o in range(co):
                if T == 8:  # up-sampling: every tap its channel
                    w[np.arange(8), rng.integers(0, ci, 8), o] = rng.choice([-1.0, 1.0], 8)
                else:
                    w[rng.integers(0, T, n), rng.integers(0, ci, n), o] = rng.choice([-1.0, 1.0], n)
        p[k] = w
    return p


def _net(G, p, base, levels, grid):
    net = G.UNet(CIN, COUT, base, levels, grid)
    net.set_params(np.concatenate([np.concatenate([p[n + ".w"].ravel(), p[n + ".b"]])
                                   for n, *_ in U.layer_spec(CIN, COUT, base, levels)]).astype(np.float32))
    return net


def _input(seed, B, grid):
    return np.random.default_rng(seed).integers(-1, 2, (B, grid, grid, grid, CIN)).astype(np.float64)


# chunks of several 64-voxel stages that cross batch entries (32^3, three
# entries: eleven stages at the fine level), 28 stages (64^3), one stage with a
# ragged end, both input halves of the decoder layers; every width of the list
@pytest.mark.parametrize("grid,B,base,levels", [(64, 1, 16, 4), (32, 3, 16, 3), (12, 3, 16, 3), (32, 3, 32, 2),
                                                (8, 3, 24, 3), (16, 1, 8, 4)])
def test_training_step_is_exact(G, grid, B, base, levels):
    p, x = _params(base + grid, base, levels), _input(grid, B, grid)
    y, cache = U.forward(p, x, levels=levels, bf=True)
    # a power of two over the count of outputs whatever the factor 3 in it
    unit = 3.0 if (B * grid) % 3 == 0 else 1.0
    if grid == 12:
        unit = 81.0
    e = unit * np.random.default_rng(1).integers(-1, 2, y.shape)
    _, dy = U.mse(y, y - e)
    ref = U.backward(p, cache, dy, levels=levels, bf=True)
    net = _net(G, p, base, levels, grid)
    assert np.array_equal(net.forward(x.astype(np.float32)), y)
    net.train_step(x.astype(np.float32), (y - e).astype(np.float32), 0.0)
    g, at = net.get_grads().astype(np.float64), 0
    for n, *_ in U.layer_spec(CIN, COUT, base, levels):
        for k in (n + ".w", n + ".b"):
            got = g[at : at + ref[k].size].reshape(ref[k].shape)
            at += ref[k].size
            assert np.array_equal(got, ref[k]), (k, np.argwhere(got != ref[k])[:4], np.max(np.abs(got - ref[k])))


# every tile plan of every layer's list, forced, with ragged tiles in x, y and z
@pytest.mark.parametrize("grid,B,base,levels", [(40, 2, 16, 4), (20, 3, 32, 3), (24, 1, 24, 3)])
def test_forward_is_exact_under_every_plan(G, grid, B, base, levels):
    p, x = _params(base + grid, base, levels), _input(grid, B, grid)
    y, _ = U.forward(p, x, levels=levels, bf=True)
    net = _net(G, p, base, levels, grid)
    most = G.gnb_unet_test_set_plan(net.h, -1)
    assert 3 <= most <= 24
    for plan in range(-1, most):
        assert G.gnb_unet_test_set_plan(net.h, plan) == most
        assert np.array_equal(net.forward(x.astype(np.float32)), y), plan


# 10^x of the remap's weights against 113-bit arithmetic: the table's entry and
# the last multiply-add round once each (2^-53 of the result), the reduction and
# the polynomial add less than a twentieth of that; outside +-290 the library's
def test_remap_exp10(G):
    import ctypes as C
    if np.finfo(np.longdouble).nmant < 100:
        pytest.skip("long double is not quadruple precision here")
    rng = np.random.default_rng(0)
    x = np.concatenate([rng.uniform(-40.0, 40.0, 60000), rng.uniform(-289.9, 289.9, 30000), np.arange(-280.0, 281.0),
                        rng.normal(size=5000) * 1e-6, np.log10(2.0) / 256.0 * np.arange(-3001.0, 3002.0, 2.0)])
    sp = np.array([0.0, 400.0, -400.0, np.inf, -np.inf, np.nan, 308.0, -320.0])
    v = np.ascontiguousarray(np.concatenate([x, sp]))
    y = np.empty_like(v)
    ptr = C.POINTER(C.c_double)
    assert G.gnb_test_exp10(v.size, v.ctypes.data_as(ptr), y.ctypes.data_as(ptr)) == G.GNB_OK
    ref = np.power(np.longdouble(10.0), x.astype(np.longdouble))
    assert np.max(np.abs(y[: x.size].astype(np.longdouble) / ref - 1)) < 2.1 * 2.0**-53
    s = y[x.size :]
    assert s[0] == 1.0 and s[1] == np.inf and s[2] == 0.0 and s[3] == np.inf and s[4] == 0.0 and np.isnan(s[5])
    assert abs(s[6] / 1e308 - 1.0) < 1e-15 and 0.0 < s[7] < 1.1e-320
