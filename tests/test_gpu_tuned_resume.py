"""A checkpoint of a handle whose kernel shapes were chosen by trial resumes bit for
bit in a handle that was never tuned: on crowded grids the two searches list a
row in different orders, and the checkpoint says which one wrote it."""
import ctypes

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    import paper_2108_01013_gb300 as dss
    from paper_2108_01013_gb300 import _native, synth
    dss.build()
    synth.build()
    return dict(dss=dss, synth=synth, lib=_native.load())


def ran(env, s, which=None):
    r = ctypes.c_int32(0)
    if which is not None:
        assert env["lib"].dss_selftest_search(s._h, which, ctypes.byref(r)) == 0
    return r.value


def state(s):
    return [v.cpu().numpy() for v in s.state().values()] + list(s.history()) + [s.stress()]


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("far", [False, True])
@pytest.mark.parametrize("search", [0, 1, 4])
def test_resume_of_a_forced_search(env, precision, far, search):
    g = env["synth"].small(4000, 0.54, 41)
    kw = dict(mu=1.0, shear_rate=5.0, precision=precision, cell_size=g["box"][0] / 5.0 * (1.0 - 1e-12), dt=1e-4)
    if far:
        kw.update(f_er=1.0, lambda_d=0.05, delta_lub=0.05)
    make = lambda: env["dss"].Suspension(g["x"], g["a"], g["box"], env["dss"].default_params(g["box"], **kw),
                                         ids=g["ids"])
    a = make()
    ran(env, a, search)
    a.step(12)
    ck = a.save()
    a.step(20)
    for other in (0, 1, 4):          # whatever the handle ran before
        b = make()
        ran(env, b, other)
        b.step(2)
        b.load(ck)
        b.step(20)
        for u, v in zip(state(a), state(b)):
            np.testing.assert_array_equal(u, v)
        b.close()
    a.close()


def test_tuned_handle_and_its_checkpoint(env):
    """dss_autotune_kernels on a crowded grid leaves the state; a checkpoint after it
    resumes alike in an untuned handle, one that is not the library's is refused."""
    g = env["synth"].small(4000, 0.54, 42)
    p = env["dss"].default_params(g["box"], shear_rate=5.0, precision="mixed",
                                  cell_size=g["box"][0] / 5.0 * (1.0 - 1e-12))
    a = env["dss"].Suspension(g["x"], g["a"], g["box"], p, ids=g["ids"])
    a.step(5)
    before = state(a)
    choice, trials = a.autotune_kernels(trial_steps=3)
    assert set(trials) == {(3, 1), (3, 4), (4, 1), (4, 4)} and choice in trials
    for u, v in zip(before, state(a)):
        np.testing.assert_array_equal(u, v)
    ck = a.save()
    a.step(10)
    b = env["dss"].Suspension(g["x"], g["a"], g["box"], p, ids=g["ids"])
    b.load(ck)
    b.step(10)
    for u, v in zip(state(a), state(b)):
        np.testing.assert_array_equal(u, v)
    for version in (0, 2, 1 | 2 << 8, 1 | 5 << 12, 1 | 1 << 16):
        bad = bytearray(ck)
        bad[8:12] = version.to_bytes(4, "little")
        with pytest.raises(env["dss"].DssError) as e:
            b.load(bytes(bad))
        assert e.value.code == -1
    a.close()
    b.close()
