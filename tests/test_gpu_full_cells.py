"""Cells of more particles than their rows of ids hold (four times the average
of the whole grid and twelve, four ids on nearly empty grids): clumps, size
classes and batches of unlike instances.  Pairs as the brute force has them,
runs of steps as single steps, and no memory beyond what the handle began
with."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    import oracle
    import paper_2108_01013_gb300 as dss
    oracle.build()
    dss.build()
    return dict(oracle=oracle, dss=dss)


def clump(n, spacing, box, seed, rest=0, a_rest=1.0):
    """n unit spheres on a jittered cubic lattice in a corner of the box, rest
    more of radius a_rest strewn over it, in random order."""
    rng = np.random.default_rng(seed)
    m = int(np.ceil(n ** (1.0 / 3.0)))
    g = np.stack(np.meshgrid(*[np.arange(m)] * 3, indexing="ij")).reshape(3, -1)[:, :n]
    x = spacing * (g + 0.5) + 0.02 * rng.standard_normal((3, n))
    x = np.concatenate([x, rng.uniform(0.0, 1.0, size=(3, rest)) * np.asarray(box)[:, None]], axis=1)
    a = np.concatenate([np.ones(n), np.full(rest, a_rest)])
    order = rng.permutation(n + rest)
    box = np.asarray(box, dtype=np.float64)
    return dict(x=x[:, order] % box[:, None], a=a[order], box=box, ids=rng.permutation(n + rest).astype(np.int32))


def want(env, g, nstep, **kw):
    po = env["oracle"].make_params(g["box"], **kw)
    return env["oracle"].pairs_bruteforce(g["x"], g["a"], g["ids"], po, env["oracle"].le_offset(po, nstep))


@pytest.mark.parametrize("case", [
    # (per cell of the whole grid, ids a row holds): a cell's fill against it
    dict(n=1500, spacing=2.05, box=(90.0, 90.0, 90.0), rest=20, a_rest=1.4),                # 0.05, 4: up to 8
    dict(n=1500, spacing=1.0, box=(60.0, 50.0, 40.0)),                                      # 0.1, 8: up to 12
    dict(n=1500, spacing=0.5, box=(40.0, 40.0, 40.0), rest=2000),                           # 0.5, 16: up to 66
    dict(n=4000, spacing=1.0, box=(110.0, 90.0, 90.0), rest=30, a_rest=9.0),                # 50, 216: up to 4000
    dict(n=1500, spacing=1.2, box=(110.0, 90.0, 90.0), rest=30, a_rest=9.0, cell_mode=1),   # size classes
])
@pytest.mark.parametrize("nstep", [0, 4321])
def test_pairs_of_full_cells(env, case, nstep):
    case = dict(case)
    extra = {k: case.pop(k) for k in ("cell_mode",) if k in case}
    g = clump(seed=17, **case)
    kw = dict(shear_rate=1.0, dt=1e-3)
    p = env["dss"].default_params(g["box"], capacity_M=1200, pair_capacity=600, **kw, **extra)
    z = np.zeros_like(g["x"])
    s = env["dss"].Suspension(g["x"], g["a"], g["box"], p, ids=g["ids"], nstep=nstep, alpha_lin=z, alpha_ang=z)
    b = s.device_bytes()
    w = want(env, g, nstep, **kw)
    for _ in range(3):
        s.neighbour_build()
        np.testing.assert_array_equal(s.pairs(), w)
    assert s.device_bytes() == b
    # the clump elsewhere: the chains of before are gone
    g["x"] = (g["x"] + 0.37 * g["box"][:, None]) % g["box"][:, None]
    s.load_state(g["x"][:, np.argsort(g["ids"])], z, z, z, z)
    h = dict(g, x=g["x"][:, np.argsort(g["ids"])], a=g["a"][np.argsort(g["ids"])], ids=np.arange(s.n, dtype=np.int32))
    s.neighbour_build()
    np.testing.assert_array_equal(s.pairs(), want(env, h, nstep, **kw))
    assert s.device_bytes() == b
    s.close()


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_runs_of_steps_over_full_cells(env, precision):
    """A clump that moves through several cells in a call, its steps begun by the
    correctors, against calls of one step."""
    g = clump(1500, 2.05, (90.0, 90.0, 90.0), 5, rest=20, a_rest=1.4)
    u = np.zeros_like(g["x"])
    u[0], u[1], u[2] = 30.0, -20.0, 25.0
    z = np.zeros_like(g["x"])
    p = env["dss"].default_params(g["box"], precision=precision, shear_rate=1.0, dt=2e-3, kn=1e3, eta0=1e-3)
    out = []
    for calls in ([8, 19, 8, 3], [1] * 38):
        s = env["dss"].Suspension(g["x"], g["a"], g["box"], p, ids=g["ids"], u=u, alpha_lin=z, alpha_ang=z)
        b = s.device_bytes()
        for k in calls:
            s.step(k)
        out.append({k: v.cpu().numpy() for k, v in s.state().items()})
        assert s.device_bytes() == b
        s.close()
    for k in out[0]:
        np.testing.assert_array_equal(out[0][k], out[1][k])
    assert np.abs(out[0]["x"] - g["x"]).max() > 1.0


def test_batch_of_unlike_instances(env):
    """One dense instance among dilute ones: the rows of ids are as long as the
    batch's average."""
    dss, orc = env["dss"], env["oracle"]
    gs = [clump(1000, 2.05, (21.0, 21.0, 21.0), 3)]
    for k in range(4):
        L = 150.0 + 10.0 * k
        gs.append(clump(300, 0.9, (L, L, L), 4 + k, rest=100))
    off = np.concatenate([[0], np.cumsum([g["a"].shape[0] for g in gs])])
    rates = [1.0, 0.5, 2.0, 1.0, 3.0]
    p = dss.default_params(dt=1e-3, capacity_M=400)
    x = np.concatenate([g["x"] for g in gs], axis=1)
    z = np.zeros_like(x)
    b = dss.Batch(x, np.concatenate([g["a"] for g in gs]), np.diff(off), [g["box"] for g in gs], rates, p, nstep=777,
                  ids=np.concatenate([g["ids"] + off[k] for k, g in enumerate(gs)]).astype(np.int32), alpha_lin=z,
                  alpha_ang=z)
    have = b.device_bytes()
    w = np.concatenate([want(env, g, 777, shear_rate=rates[k], dt=1e-3) + off[k] for k, g in enumerate(gs)])
    for _ in range(2):
        b.neighbour_build()
        np.testing.assert_array_equal(b.pairs(), w)
    assert b.device_bytes() == have
    b.close()
