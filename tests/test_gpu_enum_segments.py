"""The staged search over crowded cells (a block per segment of cells, rows
scanned in a pass of their own) against the CPU oracle's brute force, where it
can go wrong: boxes of 4 to 9 cells (every candidate exact below 7, the
shifted row as wide as the box, segments ending at the box edge), cells of
more owners than a warp holds and rows of more candidates than one tile,
batched instances of different grids, rows that overflow, pair arrays that
grow after the search."""
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
    from paper_2108_01013_gb300 import synth
    oracle.build()
    dss.build()
    synth.build()
    return dict(oracle=oracle, dss=dss, synth=synth)


def _handle(env, g, cells, nstep=0, **kw):
    """A handle whose grid has the given number of cells per axis."""
    p = env["dss"].default_params(g["box"], cell_size=g["box"][0] / cells * (1.0 - 1e-12), **kw)
    z = np.zeros_like(g["x"])
    return env["dss"].Suspension(g["x"], g["a"], g["box"], p, ids=g["ids"], nstep=nstep, alpha_lin=z, alpha_ang=z)


def _want(env, g, nstep, **kw):
    po = env["oracle"].make_params(g["box"], **kw)
    return env["oracle"].pairs_bruteforce(g["x"], g["a"], g["ids"], po, env["oracle"].le_offset(po, nstep))


@pytest.mark.parametrize("n,cells", [(600, 4), (1200, 5), (2500, 6), (2600, 7), (4500, 9), (5000, 4), (9000, 5)])
@pytest.mark.parametrize("nstep", [0, 777, 54321])
def test_segment_pairs_bit_exact(env, n, cells, nstep):
    g = env["synth"].small(n, 0.50, 900 + n)
    kw = dict(shear_rate=1.3, dt=1e-3)
    s = _handle(env, g, cells, nstep, **kw)
    assert s.counters()["ncell"] == (cells,) * 3 and n >= 4 * cells ** 3
    s.neighbour_build()
    np.testing.assert_array_equal(s.pairs(), _want(env, g, nstep, **kw))
    c = s.counters()
    rows = np.bincount(_want(env, g, nstep, **kw).reshape(-1), minlength=n)
    assert 0 < c["max_row"] <= rows.max()
    s.close()


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("forces", ["contact", "far"])
def test_segment_forces_as_on_sparse_grid(env, precision, forces):
    """The same forces on the grid that is walked owner by owner.  The rows
    differ in their order alone: the sums of at most 60 pair terms differ by
    less than 60 roundings of the particle's largest (FP64 2^-52, mixed 2^-23),
    taken relative to the largest force of the packing."""
    g = env["synth"].small(4000, 0.50, 77)
    kw = dict(shear_rate=1.0, precision=precision)
    if forces == "far":      # listed beyond the lubrication range: rows in two parts
        kw.update(f_er=10.0, lambda_d=0.05, delta_lub=0.1)
    out = []
    for cells in (5, int(g["box"][0] / (2.8 + (1.0 if forces == "far" else 0.07) + 1e-6))):
        s = _handle(env, g, cells, 31, **kw)
        F, T = s.forces()
        out.append((F.cpu().numpy(), T.cpu().numpy(), s.pairs()))
        s.close()
    np.testing.assert_array_equal(out[0][2], out[1][2])
    tol = 60 * (2.0 ** -52 if precision == "fp64" else 2.0 ** -23)
    for a, b in zip(out[0][:2], out[1][:2]):
        assert np.abs(a - b).max() <= tol * np.abs(b).max()


def test_segment_batch(env):
    """Instances of 343 to 1728 cells' worth of different boxes in one launch."""
    dss, orc = env["dss"], env["oracle"]
    gs = [env["synth"].small(n, phi, 60 + n) for n, phi in [(3000, 0.5), (900, 0.42), (5200, 0.55), (2048, 0.48)]]
    off = np.concatenate([[0], np.cumsum([g["a"].shape[0] for g in gs])])
    rates = [0.5, 3.0, 1.0, 20.0]
    p = dss.default_params(cell_size=gs[1]["box"][0] / 4.0 * (1.0 - 1e-12), dt=1e-3)
    x = np.concatenate([g["x"] for g in gs], axis=1)
    z = np.zeros_like(x)
    b = dss.Batch(x, np.concatenate([g["a"] for g in gs]), np.diff(off), [g["box"] for g in gs], rates, p, nstep=333,
                  alpha_lin=z, alpha_ang=z)
    b.neighbour_build()
    want = []
    for k, g in enumerate(gs):
        po = orc.make_params(g["box"], shear_rate=rates[k], dt=1e-3)
        want.append(orc.pairs_bruteforce(g["x"], g["a"], g["ids"], po, orc.le_offset(po, 333)) + off[k])
    np.testing.assert_array_equal(b.pairs(), np.concatenate(want))
    b.close()


@pytest.mark.parametrize("cells", [5, 0])
def test_pair_arrays_that_grow_after_the_search(env, cells):
    """A force evaluation whose pairs exceed the pair arrays lists them again:
    the same bits as with room from the start."""
    g = env["synth"].small(2000, 0.52, 5)
    cells = cells or int(g["box"][0] / 2.871)
    out = []
    for cap in (1, 32):
        s = _handle(env, g, cells, 3, pair_capacity=cap)
        F, T = s.forces()
        out.append((F.cpu().numpy(), T.cpu().numpy(), s.pairs(), s.counters()["band_checks"]))
        s.step(3)
        out[-1] += (s.state()["x"].cpu().numpy(),)
        s.close()
    for a, b in zip(*out):
        np.testing.assert_array_equal(a, b)


def test_segment_row_overflow_is_reported(env):
    g = env["synth"].small(3000, 0.55, 9)
    s = _handle(env, g, 5, 0, capacity_M=2)
    with pytest.raises(env["dss"].DssError) as e:
        s.neighbour_build()
    assert e.value.code == -3
    s.close()


def test_cells_fuller_than_their_id_rows(env):
    """Clumps of more particles per cell than the sort's rows of ids hold (four
    times the average and twelve): the order and the pairs are those of any
    other cell, before and after the host lengthens the rows."""
    rng = np.random.default_rng(3)
    n, L = 3000, 60.0
    x = rng.uniform(0.0, L, size=(3, n))
    x[:, :900] = rng.uniform(0.5, 6.5, size=(3, 900))      # ~700 in 27 of 8000 cells, up to ~60 in one
    x[:, 900:1000] = rng.uniform(31.0, 33.0, size=(3, 100))
    g = dict(x=x, a=np.ones(n), box=np.array([L, L, L]), ids=rng.permutation(n).astype(np.int32))
    kw = dict(shear_rate=1.0, dt=1e-6)
    p = env["dss"].default_params(g["box"], capacity_M=400, **kw)
    z = np.zeros_like(x)
    s = env["dss"].Suspension(x, g["a"], g["box"], p, ids=g["ids"], alpha_lin=z, alpha_ang=z, nstep=5)
    for _ in range(3):
        s.neighbour_build()
        np.testing.assert_array_equal(s.pairs(), _want(env, g, 5, **kw))
    s.close()


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("ext", [False, True])
def test_runs_of_steps_as_single_steps(env, precision, ext):
    """Steps in one call, whose correctors begin the next step, against as many
    calls of one step: the same bits, through box crossings and box offsets."""
    g = env["synth"].small(1500, 0.50, 21)
    kw = dict(mu=0.5, shear_rate=40.0, dt=1e-4, precision=precision)
    if ext:
        kw.update(wave_amp=2.0, wave_n=1, k_r=500.0)
    out = []
    for calls in ([19, 8, 3], [1] * 30):
        s = env["dss"].Suspension(g["x"], g["a"], g["box"], env["dss"].default_params(g["box"], **kw), ids=g["ids"],
                                  nstep=9990)
        for k in calls:
            s.step(k)
        c = s.counters()
        st = {k: v.cpu().numpy() for k, v in s.state().items()}
        out.append((st, s.stress(), s.images(), c["npairs"], c["ncontacts"], c["max_row"], c["band_checks"]))
        s.close()
    for k in out[0][0]:
        np.testing.assert_array_equal(out[0][0][k], out[1][0][k])
    for a, b in zip(out[0][1:], out[1][1:]):
        np.testing.assert_array_equal(a, b)


@pytest.mark.parametrize("cells", [(16, 16, 8), (17, 11, 11), (12, 13, 13), (64, 64, 63), (64, 64, 64),
                                   (65, 64, 64), (128, 64, 64), (129, 64, 64)])
def test_cell_scan_at_tile_edges(env, cells):
    """Grids of one scan tile of 2048 cells exactly, a little more and less, of
    128 tiles, of 256 (the most whose sums the histogram keeps) and a little
    more: every search, also one behind another, finds the brute force's pairs."""
    rng = np.random.default_rng(sum(cells))
    box = 3.0 * np.array(cells, dtype=np.float64)
    x = rng.uniform(0.0, 1.0, size=(3, 1500)) * box[:, None]
    d = rng.normal(size=(3, 1500))
    x = np.concatenate([x, (x + 2.03 * d / np.linalg.norm(d, axis=0)) % box[:, None]], axis=1)
    n = x.shape[1]
    g = dict(x=x, a=np.ones(n), box=box, ids=rng.permutation(n).astype(np.int32))
    p = env["dss"].default_params(box, cell_size=3.0 * (1.0 - 1e-12), capacity_M=64, shear_rate=1.0, dt=1e-6)
    z = np.zeros_like(x)
    s = env["dss"].Suspension(x, g["a"], box, p, ids=g["ids"], alpha_lin=z, alpha_ang=z, nstep=7)
    assert s.counters()["ncell"] == cells
    want = _want(env, g, 7, shear_rate=1.0, dt=1e-6)
    assert want.shape[0] > 1000
    for _ in range(3):
        s.neighbour_build()
        np.testing.assert_array_equal(s.pairs(), want)
    s.close()


@pytest.mark.parametrize("n,lam,cells", [(4000, 0.05, 5), (4000, 0.15, 4), (700, 0.05, 4)])
def test_long_rows_summed_ahead_of_the_corrector(env, n, lam, cells):
    """Forces of rows of 9 to some 100 records on a crowded grid (every such row
    becomes its sum first) as with lists by size class (rows summed in the
    corrector).  Both orders of at most 300 pair terms in FP32: they differ by
    less than 300 roundings of 2^-23 of the packing's largest force."""
    g = env["synth"].small(n, 0.50, 78)
    kw = dict(shear_rate=1.0, precision="mixed", f_er=10.0, lambda_d=lam, delta_lub=0.1)
    s = _handle(env, g, cells, 31, **kw)
    assert n >= 6 * cells ** 3
    p = env["dss"].default_params(g["box"], cell_mode=1, **kw)
    z = np.zeros_like(g["x"])
    c = env["dss"].Suspension(g["x"], g["a"], g["box"], p, ids=g["ids"], nstep=31, alpha_lin=z, alpha_ang=z)
    out = []
    for h in (s, c):
        F, T = h.forces()
        out.append((F.cpu().numpy(), T.cpu().numpy(), h.pairs()))
    np.testing.assert_array_equal(out[0][2], out[1][2])
    assert np.bincount(out[0][2].reshape(-1)).max() > 9
    for a, b in zip(out[0][:2], out[1][:2]):
        assert np.abs(a - b).max() <= 300 * 2.0 ** -23 * np.abs(b).max()
    s.close()
    c.close()


@pytest.mark.parametrize("cells", [(4, 3, 3), (4, 4, 3), (5, 3, 4), (6, 5, 3), (4, 5, 6)])
@pytest.mark.parametrize("nstep", [0, 250, 999, 54321])
def test_narrow_boxes_pair_by_the_nearest_image(env, cells, nstep):
    """Boxes of three to six cells, where the stencil meets separations beyond
    half the box: the pairs of the nearest images, as the brute force has them.
    Random centres, half of them on multiples of half a cell."""
    rng = np.random.default_rng(sum(cells) + nstep)
    edge = 2.9
    box = edge * np.array(cells, dtype=np.float64)
    n = 12 * int(np.prod(cells))
    x = rng.uniform(0.0, 1.0, size=(3, n)) * box[:, None]
    x[:, ::2] = np.round(x[:, ::2] / (0.5 * edge)) * (0.5 * edge) % box[:, None]
    x[:, ::2] += rng.uniform(0.0, 1e-3, size=x[:, ::2].shape)
    g = dict(x=x, a=rng.choice([1.0, 1.4], size=n), box=box, ids=rng.permutation(n).astype(np.int32))
    kw = dict(shear_rate=1.3, dt=1e-3)
    p = env["dss"].default_params(box, cell_size=edge * (1.0 - 1e-12), capacity_M=400, **kw)
    z = np.zeros_like(x)
    s = env["dss"].Suspension(x, g["a"], box, p, ids=g["ids"], nstep=nstep, alpha_lin=z, alpha_ang=z)
    assert s.counters()["ncell"] == cells
    s.neighbour_build()
    np.testing.assert_array_equal(s.pairs(), _want(env, g, nstep, **kw))
    s.close()
