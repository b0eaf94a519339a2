"""Steps by graphs of 8, 4, 2 and 1: the graphs of 4 and 2 steps are captured when
they are wanted a second time, so every run length comes twice and more here, from
either buffer role, and once more after the graphs have been dropped."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

RUNS = [7, 7, 6, 6, 3, 3, 1, 7, 15, 14, 2, 4, 4, 2, 8, 5]


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


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("kind", ["contact", "extended", "crowded", "batch"])
def test_every_graph_as_single_steps(env, precision, kind):
    dss = env["dss"]
    g = env["synth"].small(1500, 0.50, 21)
    kw = dict(mu=0.5, shear_rate=40.0, dt=1e-4, precision=precision)
    if kind == "extended":
        kw.update(wave_amp=2.0, wave_n=1, k_r=500.0)
    if kind == "crowded":      # long rows: no step begins the next one
        kw.update(f_er=1.0, lambda_d=0.1, delta_lub=0.1, cell_size=g["box"][0] / 4.0 * (1.0 - 1e-12))
    out = []
    for calls in (RUNS, [1] * sum(RUNS)):
        p = dss.default_params(g["box"], **kw)
        if kind == "batch":
            s = dss.Batch(np.concatenate([g["x"]] * 2, axis=1), np.concatenate([g["a"]] * 2), [1500, 1500], [g["box"]] * 2,
                          [40.0, 10.0], p, nstep=9990)
        else:
            s = dss.Suspension(g["x"], g["a"], g["box"], p, ids=g["ids"], nstep=9990)
        for k, c in enumerate(calls):
            if len(calls) == len(RUNS) and k == 8:      # the graphs anew, from wherever the roles are
                s.set_profiling(True)
                s.step(1)
                s.set_profiling(False)
                c -= 1
            s.step(c)
        c = s.counters()
        st = {k: v.cpu().numpy() for k, v in s.state().items()}
        sig = s.batch_stress()[:2] if kind == "batch" else (s.stress(), s.rheology(mean=True))
        out.append((st, sig[0], sig[1], s.images(), c["npairs"], c["ncontacts"], c["max_row"], c["band_checks"]))
        assert c["steps_done"] == sum(RUNS)
        s.close()
    for k in out[0][0]:
        np.testing.assert_array_equal(out[0][0][k], out[1][0][k])
    for a, b in zip(out[0][1:], out[1][1:]):
        np.testing.assert_array_equal(a, b)
