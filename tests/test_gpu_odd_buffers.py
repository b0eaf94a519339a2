"""Device buffers at odd addresses: forces, state and host-owned steps as with
aligned ones (they go through the library's own arrays and a copy)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def test_buffers_at_odd_addresses():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    import paper_2108_01013_gb300 as dss
    from paper_2108_01013_gb300 import _native as nat, synth
    dss.build()
    synth.build()
    g = synth.small(700, 0.5, 4)
    n = g["a"].size
    lib = nat.load()
    raw = [torch.zeros(24 * n + 8, dtype=torch.uint8, device="cuda") for _ in range(5)]

    def read(t):
        torch.cuda.synchronize()
        return np.frombuffer(t.cpu().numpy()[4:4 + 24 * n].tobytes()).reshape(3, n)

    out = []
    for _ in range(2):
        s = dss.Suspension(g["x"], g["a"], g["box"], dss.default_params(g["box"], dt=1e-5), ids=g["ids"])
        s.step(2)
        if not out:
            F, T = s.forces()
            st = s.state()
            have = [F, T] + [st[k] for k in ("x", "u", "w", "al", "aw")]
            have = [t.cpu().numpy() for t in have]
            s.step(1)
            out.append(have + [s.state()["x"].cpu().numpy()])
        else:
            p = [t.data_ptr() + 4 for t in raw]
            assert lib.dss_force_eval(s._h, p[0], p[1]) == 0
            have = [read(raw[0]), read(raw[1])]
            assert lib.dss_get_state(s._h, *p) == 0
            have += [read(t) for t in raw]
            assert lib.dss_load_state(s._h, *p) == 0
            s.step(1)
            out.append(have + [s.state()["x"].cpu().numpy()])
        s.close()
    for a, b in zip(*out):
        np.testing.assert_array_equal(a, b)
