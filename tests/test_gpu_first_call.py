"""The first call of a circuit makes and uploads the plan of its staged passes: without waiting for work
queued elsewhere, and without breaking a capture that runs on another stream."""
import time

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


def circuit(n, seed, count=60):
    rng = np.random.default_rng(seed)
    return [wl.random_gate(n, int(rng.integers(1, 4)), rng) for _ in range(count)]


def check(B, st, gates, f):
    got, n = st.store(), st.n
    # one fused gate's error on a unit vector is at most (2^(k+1) + 2) 2^-24
    tol = sum((2 ** (B.sv_fused_get_info(f, i)["k"] + 1) + 2) * 2.0 ** -24 for i in range(B.sv_fused_count(f)))
    assert oracle.l2_error(oracle.run_circuit(n, gates, 0), got) <= tol


@pytest.mark.parametrize("lazy", [False, True])
def test_does_not_wait_for_queued_work(B, lazy):
    import torch
    from paper_2602_09604_gb300.state import DeviceState
    n = 14
    s = torch.cuda.Stream()
    st = DeviceState(n, stream=s)
    circuits = [circuit(n, i) for i in range(3)]
    fused = [B.sv_fuse_circuit(g, n, max_k=3) for g in circuits]

    def step(f):
        if lazy:
            B.sv_init_apply(st.h, 0, f)
        else:
            st.init(0)
            st.apply(f)

    step(fused[0])   # the state's own buffers, the library's staging buffer and stream
    torch.cuda.synchronize()
    done = torch.cuda.Event()
    torch.cuda._sleep(1_500_000_000)   # about 0.8 s on the legacy stream
    done.record()
    began = time.monotonic()
    step(fused[1])
    took = time.monotonic() - began
    assert not done.query() and took < 0.3, took
    check(B, st, circuits[1], fused[1])
    torch.cuda.synchronize()
    for f in fused:
        B.sv_fused_free(f)
    st.free()


def test_during_another_streams_capture(B):
    import torch
    from paper_2602_09604_gb300.state import DeviceState
    n = 14
    a, b = torch.cuda.Stream(), torch.cuda.Stream()
    sa, sb = DeviceState(n, stream=a), DeviceState(n, stream=b)
    gates = [circuit(n, 10), circuit(n, 11)]
    fa, fb = (B.sv_fuse_circuit(g, n, max_k=3) for g in gates)
    sa.init(0)
    sa.apply(fa)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.stream(a):
        graph.capture_begin(capture_error_mode="global")
        sa.init(0)
        sa.apply(fa)
        sb.init(0)
        sb.apply(fb)   # its first call, on a stream that is not captured
        graph.capture_end()
        graph.replay()
    torch.cuda.synchronize()
    check(B, sa, gates[0], fa)
    check(B, sb, gates[1], fb)
    for f in (fa, fb):
        B.sv_fused_free(f)
    sa.free()
    sb.free()
