"""The two searches of the enumeration, each forced on the same handle: the walk by
owner (k_enumerate) and the staged search (k_enumerate_seg).  The built-in rule
gives small single systems and crowded grids to the staged one, so that most of
the small cases elsewhere run it alone.  Pairs against the brute force: random
packings, centres near the cutoff by ulps, particles along the sheared boundary,
narrow boxes, radii spread over a factor of three; forces of either as the
other's."""
import ctypes

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

WALK, STAGED = 1, 4


@pytest.fixture(scope="module")
def env():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    import oracle
    import paper_2108_01013_gb300 as dss
    from paper_2108_01013_gb300 import _native, synth
    oracle.build()
    dss.build()
    synth.build()
    return dict(oracle=oracle, dss=dss, synth=synth, lib=_native.load())


def force(env, s, which):
    ran = ctypes.c_int32(0)
    assert env["lib"].dss_selftest_search(s._h, which, ctypes.byref(ran)) == 0
    assert ran.value == which


def check_pairs(env, g, nsteps, cell_size=0.0, **kw):
    p = env["dss"].default_params(g["box"], cell_size=cell_size, capacity_M=400, **kw)
    po = env["oracle"].make_params(g["box"], **kw)
    z = np.zeros_like(g["x"])
    total = 0
    for nstep in nsteps:
        s = env["dss"].Suspension(g["x"], g["a"], g["box"], p, ids=g["ids"], nstep=nstep, alpha_lin=z, alpha_ang=z)
        want = env["oracle"].pairs_bruteforce(g["x"], g["a"], g["ids"], po, env["oracle"].le_offset(po, nstep))
        for which in (WALK, STAGED, WALK):
            force(env, s, which)
            s.neighbour_build()
            np.testing.assert_array_equal(s.pairs(), want)
        total += len(want)
        s.close()
    return total


@pytest.mark.parametrize("n,phi,mode,delta", [(300, 0.45, 0, 0.05), (777, 0.55, 0, 0.05), (1501, 0.52, 1, 0.08),
                                              (2048, 0.40, 0, 0.25)])
def test_random_packings(env, n, phi, mode, delta):
    g = env["synth"].small(n, phi, n)
    assert check_pairs(env, g, (0, 31, 12345, 987654), lub_cutoff_mode=mode, delta_lub=delta, shear_rate=1.3,
                       dt=1e-3) > n


@pytest.mark.parametrize("lam", [0.05, 0.002])
def test_wider_listing_ranges(env, lam):
    """Electro-chemical ranges beyond every lubrication range, and between the
    smallest and the largest."""
    g = env["synth"].small(1200, 0.48, 3)
    check_pairs(env, g, (0, 4567), shear_rate=1.3, dt=1e-3, f_er=10.0, lambda_d=lam, delta_lub=0.035)


def test_spread_radii_along_the_sheared_boundary(env):
    rng = np.random.default_rng(9)
    g = env["synth"].generate(env["synth"].Spec("poly", 1200, 0.45, radii="loguniform", a_min=1.0, a_max=3.0, seed=21))
    g = dict(x=g["x"].copy(), a=g["a"], ids=g["ids"], box=g["box"])
    k = rng.choice(1200, size=400, replace=False)
    g["x"][1, k[:200]] = rng.uniform(0, 2.0, size=200)
    g["x"][1, k[200:]] = g["box"][1] - rng.uniform(1e-9, 2.0, size=200)
    check_pairs(env, g, (0, 7, 333, 1001, 5555), shear_rate=0.9, dt=1e-2)


def test_pairs_near_the_cutoff(env):
    rng = np.random.default_rng(4)
    box = np.array([30.0, 30.0, 30.0])
    pts, rad = [], []
    for t in range(80):
        c = rng.uniform(0, 30, size=3)
        u = rng.normal(size=3)
        ai, aj = (1.0, 1.4) if t % 2 else (1.4, 1.4)
        r = (ai + aj) * 1.025 * (1 + rng.choice([-1, 1]) * rng.uniform(0, 4e-16))
        pts += [c, c + r * u / np.linalg.norm(u)]
        rad += [ai, aj]
    x = np.mod(np.array(pts).T, box[:, None])
    x[x >= 30.0] = 0.0
    check_pairs(env, dict(x=x, a=np.array(rad), box=box, ids=np.arange(160, dtype=np.int32)), (0,), shear_rate=0.0)


@pytest.mark.parametrize("cells", [(4, 3, 3), (4, 4, 3), (5, 3, 4), (6, 5, 3), (7, 4, 5)])
def test_narrow_boxes(env, cells):
    rng = np.random.default_rng(sum(cells))
    edge = 2.9
    box = edge * np.array(cells, dtype=np.float64)
    n = 12 * int(np.prod(cells))
    x = rng.uniform(0.0, 1.0, size=(3, n)) * box[:, None]
    x[:, ::2] = np.round(x[:, ::2] / (0.5 * edge)) * (0.5 * edge) % box[:, None]
    x[:, ::2] += rng.uniform(0.0, 1e-3, size=x[:, ::2].shape)
    g = dict(x=x, a=rng.choice([1.0, 1.4], size=n), box=box, ids=rng.permutation(n).astype(np.int32))
    check_pairs(env, g, (0, 250, 999, 54321), cell_size=edge * (1.0 - 1e-12), shear_rate=1.3, dt=1e-3)


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("far", [False, True])
def test_forces_alike(env, precision, far):
    """Rows differ in their order alone: sums of at most 60 pair terms differ by less
    than 60 roundings of the packing's largest force."""
    g = env["synth"].small(4000, 0.50, 77)
    kw = dict(f_er=10.0, lambda_d=0.05, delta_lub=0.1) if far else {}
    p = env["dss"].default_params(g["box"], precision=precision, cell_size=g["box"][0] / 6.0 * (1.0 - 1e-12), **kw)
    z = np.zeros_like(g["x"])
    s = env["dss"].Suspension(g["x"], g["a"], g["box"], p, ids=g["ids"], nstep=31, alpha_lin=z, alpha_ang=z)
    out = []
    for which in (WALK, STAGED):
        force(env, s, which)
        out.append([t.cpu().numpy() for t in s.forces()])
    tol = 60 * (2.0 ** -52 if precision == "fp64" else 2.0 ** -23)
    for a, b in zip(*out):
        assert np.abs(a - b).max() <= tol * np.abs(b).max()
    s.close()


def test_batch(env):
    gs = [env["synth"].small(n, phi, 60 + n) for n, phi in [(3000, 0.5), (900, 0.42), (2048, 0.48)]]
    off = np.concatenate([[0], np.cumsum([g["a"].shape[0] for g in gs])])
    rates = [0.5, 3.0, 1.0]
    x = np.concatenate([g["x"] for g in gs], axis=1)
    z = np.zeros_like(x)
    b = env["dss"].Batch(x, np.concatenate([g["a"] for g in gs]), np.diff(off), [g["box"] for g in gs], rates,
                         env["dss"].default_params(dt=1e-3), nstep=333, alpha_lin=z, alpha_ang=z)
    want = []
    for k, g in enumerate(gs):
        po = env["oracle"].make_params(g["box"], shear_rate=rates[k], dt=1e-3)
        want.append(env["oracle"].pairs_bruteforce(g["x"], g["a"], g["ids"], po, env["oracle"].le_offset(po, 333)) + off[k])
    for which in (WALK, STAGED, WALK):
        force(env, b, which)
        b.neighbour_build()
        np.testing.assert_array_equal(b.pairs(), np.concatenate(want))
    b.close()


def test_refused(env):
    g = env["synth"].small(300, 0.45, 1)
    s = env["dss"].Suspension(g["x"], g["a"], g["box"], env["dss"].default_params(g["box"]))
    assert env["lib"].dss_selftest_search(s._h, 3, None) == -1
    assert env["lib"].dss_selftest_search(None, 1, None) == -1
    s.step(2)
    s.close()
