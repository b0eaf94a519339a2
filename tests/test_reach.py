"""Which caller buffers a kernel accesses in place: aligned memory of the handle's
own device.  Memory of another device and odd addresses go through copies."""
import pytest

HOST, DEVICE, MANAGED, UNREGISTERED = 1, 2, 3, 0     # cudaMemoryType


@pytest.fixture(scope="module")
def reach():
    from paper_2108_01013_gb300 import _native
    _native.build()
    return _native.load().dss_selftest_reach


@pytest.mark.parametrize("mine", [0, 1, 7])
@pytest.mark.parametrize("theirs", [0, 1, 7])
def test_memory_of_the_same_device_alone(reach, mine, theirs):
    assert reach(DEVICE, theirs, mine, 0x7f0000001000) == (1 if mine == theirs else 0)


@pytest.mark.parametrize("kind", [HOST, MANAGED, UNREGISTERED])
def test_other_memory(reach, kind):
    assert reach(kind, 0, 0, 0x7f0000001000) == 0


@pytest.mark.parametrize("odd", [1, 2, 4, 7])
def test_alignment(reach, odd):
    assert reach(DEVICE, 0, 0, 0x7f0000001000 + odd) == 0
    assert reach(DEVICE, 0, 0, 0x7f0000001000 + 8 * odd) == 1
