"""Fused circuits freed while captured graphs of their staged passes, or launches made before a
capture, still need the passes' images: the graph keeps them, and sv_fused_free waits for the launches."""
import numpy as np
import pytest

import oracle
from paper_2602_09604_gb300 import build as libbuild
from paper_2602_09604_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    libbuild.build()
    import torch
    assert torch.cuda.is_available()
    from paper_2602_09604_gb300 import binding
    return binding


def circuit(n, seed, count=80):
    rng = np.random.default_rng(seed)
    return [wl.random_gate(n, int(rng.integers(1, 4)), rng) for _ in range(count)]


def fuse(B, n, seed):
    return B.sv_fuse_circuit(circuit(n, seed), n, max_k=3)


def others(B, n, count=12):
    """Circuits of the same size, applied: their images take the buffers that the cache has."""
    from paper_2602_09604_gb300.state import DeviceState
    st = DeviceState(n)
    kept = [fuse(B, n, 100 + i) for i in range(count)]
    for f in kept:
        st.init(0)
        st.apply(f)
    st.stream.synchronize()
    st.free()
    return kept


# one gate's error on a unit vector is at most (2^(k+1) + 2) 2^-24; both routes make it
def bound(B, f):
    return 2 * sum((2 ** (B.sv_fused_get_info(f, i)["k"] + 1) + 2) * 2.0 ** -24 for i in range(B.sv_fused_count(f)))


@pytest.mark.parametrize("lazy", [False, True])
@pytest.mark.parametrize("n", [13, 20])
def test_graph_replayed_after_its_circuit_is_freed(B, n, lazy):
    import torch
    from paper_2602_09604_gb300.state import DeviceState
    f = fuse(B, n, 7)
    tol = bound(B, f)
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        st = DeviceState(n, stream=s)
        B.sv_init_apply(st.h, 5, f, timings=True)
        want = st.store()
        step = (lambda: B.sv_init_apply(st.h, 5, f)) if lazy else (lambda: st.apply(f))
        step()   # makes the plan (and the small state of a lazy start)
        s.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=s):
            step()
        B.sv_fused_free(f)
        kept = others(B, n)
        for _ in range(2):
            st.init(5)
            graph.replay()
            s.synchronize()
            assert oracle.l2_error(want.astype(np.complex128), st.store()) <= tol
        del graph
    kept += others(B, n)   # the graph's buffer is the cache's again
    for f in kept:
        B.sv_fused_free(f)
    st.free()


def test_free_waits_for_launches_made_before_a_capture(B):
    import torch
    from paper_2602_09604_gb300.state import DeviceState
    n = 24
    f = fuse(B, n, 9)
    tol = bound(B, f)
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        st = DeviceState(n, stream=s)
        other = DeviceState(n, stream=s)
        other.init(0)
        st.init(3)
        st.apply(f, timings=True)
        want = st.store()
        st.apply(f)
        st.init(3)
        s.synchronize()
        st.apply(f)   # a few milliseconds, still running below
        graph = torch.cuda.CUDAGraph()
        graph.capture_begin(capture_error_mode="thread_local")
        other.apply(f)
        graph.capture_end()
        B.sv_fused_free(f)
        kept = others(B, n)
        s.synchronize()
        assert oracle.l2_error(want.astype(np.complex128), st.store()) <= tol
    for f in kept:
        B.sv_fused_free(f)
    st.free()
    other.free()
