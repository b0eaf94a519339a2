"""Orders that the step's kernels have to state in their source, since no test on
the GPU can be relied on to show their absence."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2108_01013_gb300", "csrc")


def source(name):
    text = open(os.path.join(CSRC, name)).read()
    return re.sub(r"//[^\n]*", "", text)


def kernels():
    """{name: body} of every __global__ function."""
    out = {}
    for name in sorted(os.listdir(CSRC)):
        text = source(name)
        for m in re.finditer(r"__global__[^;{]*?\b(k_\w+)\s*\(", text):
            i = text.index("{", m.end())
            depth, j = 1, i + 1
            while depth:
                depth += {"{": 1, "}": -1}.get(text[j], 0)
                j += 1
            out[m.group(1)] = text[i + 1:j - 1]
    return out


ALL = kernels()


def test_error_read_alike_by_a_warp_where_blocks_may_set_it():
    """The kernels that raise errors of their own (a full row of partner records,
    sums that are not finite) and vote or shuffle over full warps afterwards."""
    for k in ("k_pairs_pb", "k_gather"):
        head = ALL[k][:1600]
        assert "warp_err(st)" in head
        assert not re.search(r"[^_]dev_err\(st\)\s*(\)|!=)", head.split("warp_err")[0]), k


def test_kernels_wait_before_they_read():
    """Every kernel that looks at the step's error word starts by waiting for its
    predecessor (programmatic dependent launch): first statement but for shared
    arrays and names."""
    seen = 0
    for k, body in ALL.items():
        if not re.search(r"dev_err\(|warp_err\(", body):
            continue
        head = body.split("dep_wait();")[0]
        assert "dep_wait();" in body, k
        assert not re.sub(r"(__shared__|constexpr|using)[^;]*;", "", head).strip(), (k, head)
        seen += 1
    assert seen >= 10


def test_loads_in_assembly_stay_behind_the_wait():
    """A load written in assembly is not moved across the wait only when it is
    volatile, as the wait is."""
    loads = 0
    for name in sorted(os.listdir(CSRC)):
        for m in re.finditer(r"\basm\b(\s+volatile)?\s*\(\s*\"ld\.", source(name)):
            loads += 1
            assert m.group(1), (name, source(name)[m.start():m.start() + 60])
    assert loads >= 3


def test_profiled_kernels_exist():
    """The names that the per-kernel times go by are those of kernels in the sources
    (or begin theirs), and the byte tables of the benchmark go by the same."""
    import bench
    from paper_2108_01013_gb300 import _native
    _native.build()
    lib = _native.load()
    names = [lib.dss_profile_name(k).decode() for k in range(_native.PROF_KERNELS)]
    assert names == list(bench.METHOD_BYTES) == list(bench.IMPL_BYTES)
    for name in names:
        assert any(k.startswith(name) for k in ALL), name
    # a single step launches each once: the headline's count
    assert bench.KERNELS_PER_STEP == len(names)
