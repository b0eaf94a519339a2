"""The staged search where a few cells hold most of the particles (segregated
sizes): owners beyond a segment's own blocks are shared out.  Pairs as the brute
force has them, and no block left to search a full cell alone."""
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


def segregated(n, spacing, box, seed, large, a_large=9.0, corner=(0.0, 0.0, 0.0)):
    """n unit spheres on a jittered cubic lattice from a corner on, a few large
    ones strewn over the box, in random order."""
    rng = np.random.default_rng(seed)
    box = np.asarray(box, dtype=np.float64)
    m = int(np.ceil(n ** (1.0 / 3.0)))
    g = np.stack(np.meshgrid(*[np.arange(m)] * 3, indexing="ij")).reshape(3, -1)[:, :n]
    x = np.asarray(corner)[:, None] + spacing * (g + 0.5) + 0.02 * rng.standard_normal((3, n))
    x = np.concatenate([x, rng.uniform(0.0, 1.0, size=(3, large)) * box[:, None]], axis=1)
    a = np.concatenate([np.ones(n), np.full(large, a_large)])
    order = rng.permutation(n + large)
    return dict(x=x[:, order] % box[:, None], a=a[order], box=box, ids=rng.permutation(n + large).astype(np.int32))


def want(env, g, nstep, **kw):
    po = env["oracle"].make_params(g["box"], **kw)
    return env["oracle"].pairs_bruteforce(g["x"], g["a"], g["ids"], po, env["oracle"].le_offset(po, nstep))


# a segment's own blocks take all owners up to 224 beyond 32 a block, of a longer
# one 32 a block (and on to a multiple of 32 in the sorted order)
@pytest.mark.parametrize("n,spacing,box,large", [
    (600, 2.3, (110.0, 90.0, 90.0), 20),      # 8 a cell: 600 in one
    (2500, 2.05, (90.0, 90.0, 90.0), 10),     # 39 a cell, two blocks each: up to 1100 in one
    (6000, 2.05, (170.0, 130.0, 130.0), 30),  # several long segments in a row
    (256, 1.0, (110.0, 90.0, 90.0), 20),      # as long as a segment's own blocks take, and one more
    (257, 1.0, (110.0, 90.0, 90.0), 20),
])
@pytest.mark.parametrize("corner,nstep", [((0.0, 0.0, 0.0), 0), ((35.0, 80.0, 71.0), 4321)])
@pytest.mark.parametrize("forces", ["contact", "far"])
def test_pairs_of_segregated_sizes(env, n, spacing, box, large, corner, nstep, forces):
    g = segregated(n, spacing, box, n, large, corner=corner)
    kw = dict(shear_rate=1.0, dt=1e-3)
    if forces == "far":
        kw.update(f_er=10.0, lambda_d=0.01, delta_lub=0.05)
    p = env["dss"].default_params(g["box"], capacity_M=600, **kw)
    z = np.zeros_like(g["x"])
    s = env["dss"].Suspension(g["x"], g["a"], g["box"], p, ids=g["ids"], nstep=nstep, alpha_lin=z, alpha_ang=z)
    w = want(env, g, nstep, **kw)
    for _ in range(2):
        s.neighbour_build()
        np.testing.assert_array_equal(s.pairs(), w)
    s.close()


def test_batch_of_segregated_instances(env):
    dss = env["dss"]
    gs = [segregated(n, 2.1, (L, 90.0, 90.0), n, 12, corner=(10.0 * k, 40.0, 5.0))
          for k, (n, L) in enumerate([(2000, 90.0), (700, 110.0), (1500, 100.0)])]
    off = np.concatenate([[0], np.cumsum([g["a"].shape[0] for g in gs])])
    rates = [1.0, 2.0, 0.5]
    p = dss.default_params(dt=1e-3, capacity_M=600)
    x = np.concatenate([g["x"] for g in gs], axis=1)
    z = np.zeros_like(x)
    b = dss.Batch(x, np.concatenate([g["a"] for g in gs]), np.diff(off), [g["box"] for g in gs], rates, p, nstep=777,
                  ids=np.concatenate([g["ids"] + off[k] for k, g in enumerate(gs)]).astype(np.int32), alpha_lin=z,
                  alpha_ang=z)
    b.neighbour_build()
    np.testing.assert_array_equal(b.pairs(), np.concatenate(
        [want(env, g, 777, shear_rate=rates[k], dt=1e-3) + off[k] for k, g in enumerate(gs)]))
    b.close()


def test_search_of_full_cells_is_shared(env):
    """20,000 small spheres, a thousand to a cell of 512 cells: 4.0 ms when a cell's
    owners beyond its average fall to one block, 0.6 ms when every owner is
    walked by a thread."""
    g = segregated(20000, 2.06, (168.1, 168.1, 168.1), 3, 60, a_large=10.0)
    p = env["dss"].default_params(g["box"], capacity_M=800, dt=1e-7, precision="mixed", kn=1.0)
    z = np.zeros_like(g["x"])
    s = env["dss"].Suspension(g["x"], g["a"], g["box"], p, ids=g["ids"], alpha_lin=z, alpha_ang=z)
    s.step(2)
    s.set_profiling(True)
    s.step(4)
    ms, steps = s.profile()
    assert ms["k_enumerate"] / steps < 1.5
    s.close()
