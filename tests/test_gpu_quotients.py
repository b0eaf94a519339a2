"""The FP64 quotients that the kernels take from a reciprocal: the corrector's
accelerations (a / b, the rounded quotient) and a pair's 1/r, 1/S and 1/(gap +
eps) from one reciprocal, which the force pass and its reverse share."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _run(a, b, c):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    import paper_2108_01013_gb300 as dss
    from paper_2108_01013_gb300 import _native
    dss.build()
    n = a.size
    d = [torch.from_numpy(v).cuda() for v in (a, b, c)]
    q, r = torch.empty(n, dtype=torch.float64, device="cuda"), torch.empty(3 * n, dtype=torch.float64, device="cuda")
    rc = _native.load().dss_selftest_quotients(*[t.data_ptr() for t in d], n, q.data_ptr(), r.data_ptr(), None)
    assert rc == 0
    return q.cpu().numpy(), r.cpu().numpy().reshape(3, n)


def _values(n, seed):
    rng = np.random.default_rng(seed)
    return np.exp2(rng.uniform(-60.0, 60.0, size=n)) * rng.uniform(1.0, 2.0, size=n)


def test_quotient_is_the_rounded_one():
    a, b = _values(400000, 1), _values(400000, 2)
    # significands that end a binade, of ones alone, equal and next to each other
    edge = np.array([1.0, 1.0 + 2.0 ** -52, 2.0 - 2.0 ** -52, 1.5, 3.0, 4.0 / 3.0, 5.0 / 3.0, np.pi, 2.0 - 2.0 ** -51])
    a = np.concatenate([a, np.repeat(edge, edge.size), -a[:1000], np.zeros(1)])
    b = np.concatenate([b, np.tile(edge, edge.size), b[:1000], np.ones(1)])
    q, _ = _run(a, b, np.ones_like(a))
    np.testing.assert_array_equal(q, a / b)


def test_reciprocals_of_a_pair():
    """1/r and S/num after their correction lie within a rounding and a half of
    the exact quotients (2^-53 each: the correction's own rounding, and less than
    half of one left by it), 1/S, uncorrected, within six roundings."""
    rng = np.random.default_rng(3)
    n = 400000
    S = rng.uniform(0.4, 20.0, size=n)
    gap = np.where(rng.random(n) < 0.3, 0.0, np.exp2(rng.uniform(-40.0, 1.0, size=n)))
    r = S * (1.0 + 0.5 * gap) * (1.0 - 1e-3 * (gap == 0.0))
    num = S * (gap + np.where(rng.random(n) < 0.5, 1e-3, 1e-6))
    _, q = _run(r, S, num)
    ld = np.longdouble
    for k, (have, exact, most) in enumerate(zip(q, (1 / r.astype(ld), 1 / S.astype(ld), S.astype(ld) / num),
                                                (1.5, 6.0, 1.5))):
        assert np.abs(have / exact - 1).max() <= most * 2.0 ** -53 * (1.0 + 1e-6), k
