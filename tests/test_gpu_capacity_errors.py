"""Which capacity an evaluation exceeded: pair arrays that are too short are
grown and the evaluation done again; a row of more partners than M is reported,
also on a handle that has listed more pairs before than its arrays hold now."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    import paper_2108_01013_gb300 as dss
    from paper_2108_01013_gb300 import synth
    dss.build()
    synth.build()
    return dict(dss=dss, synth=synth)


@pytest.mark.parametrize("call", ["forces", "step"])
def test_row_overflow_after_more_pairs_than_the_arrays_now_hold(env, call):
    dss = env["dss"]
    g = env["synth"].small(2000, 0.52, 5)
    z = np.zeros_like(g["x"])
    p = dss.default_params(g["box"], pair_capacity=1, capacity_M=14, dt=1e-6)
    s = dss.Suspension(g["x"], g["a"], g["box"], p, ids=g["ids"], alpha_lin=z, alpha_ang=z)
    s.forces()
    if call == "step":
        s.step(2)
    assert s.counters()["npairs"] > 2 * s.n      # the arrays start at one pair a particle
    # smaller radii: the buffers are made anew, as long as at first; few pairs,
    # but thirty spheres about one point, rows of up to 29
    rng = np.random.default_rng(8)
    x = rng.uniform(0.0, 1.0, size=(3, s.n)) * g["box"][:, None]
    x[:, :30] = 0.5 * g["box"][:, None] + rng.uniform(-0.01, 0.01, size=(3, 30))
    a = np.full(s.n, 0.3)
    a[30] = 1.4
    bytes_before = s.device_bytes()
    s.set_state(x, a, alpha_lin=z, alpha_ang=z)
    assert s.device_bytes() != bytes_before
    with pytest.raises(dss.DssError) as e:
        s.forces() if call == "forces" else s.step(3)
    assert e.value.code == -3
    # the handle goes on with a state that fits
    x[:, :30] = rng.uniform(0.0, 1.0, size=(3, 30)) * g["box"][:, None]
    s.set_state(x, a, alpha_lin=z, alpha_ang=z)
    F, _ = s.forces()
    assert np.isfinite(F.cpu().numpy()).all()
    s.close()


def test_pair_arrays_still_grow(env):
    """Both growths in one handle: an evaluation's and a step's."""
    dss = env["dss"]
    g = env["synth"].small(2000, 0.52, 5)
    out = []
    for cap in (1, 32):
        s = dss.Suspension(g["x"], g["a"], g["box"], dss.default_params(g["box"], pair_capacity=cap, dt=1e-6),
                           ids=g["ids"])
        F, T = s.forces()
        s.step(3)
        out.append((F.cpu().numpy(), T.cpu().numpy(), s.state()["x"].cpu().numpy()))
        s.close()
    for a, b in zip(*out):
        np.testing.assert_array_equal(a, b)


@pytest.mark.parametrize("n", [3000, 400_000])
def test_pairs_after_rows_that_overflow(env, n):
    """Reading a list whose build was refused is safe: what it gives are pairs of
    ids, no more than the rows hold, and the handle goes on."""
    dss = env["dss"]
    rng = np.random.default_rng(n)
    L = (n * 12.0) ** (1.0 / 3.0)
    x = rng.uniform(0.0, L, size=(3, n))
    z = np.zeros_like(x)
    s = dss.Suspension(x, np.ones(n), [L] * 3, dss.default_params(capacity_M=40), alpha_lin=z, alpha_ang=z)
    s.neighbour_build()
    full = s.pairs()
    s.close()
    s = dss.Suspension(x, np.ones(n), [L] * 3, dss.default_params(capacity_M=1), alpha_lin=z, alpha_ang=z)
    for _ in range(3):
        with pytest.raises(dss.DssError) as e:
            s.neighbour_build()
        assert e.value.code == -3
        p = s.pairs()
        assert len(p) <= n and (p >= 0).all() and (p < n).all() and (p[:, 0] < p[:, 1]).all()
    assert len(full) > n
    s.close()
