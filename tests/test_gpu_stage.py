"""Staged passes (several fused gates per pass through shared-memory tiles, taken by calls without
timing records) against the oracle and against the one-launch-per-gate route (calls with timing
records): tile edges (states smaller than, equal to and just above one tile), every fused size, kept
controls inside and outside a tile, starts through sv_init_apply, and circuits with tensor-core
gates, whose passes keep the circuit's order and so give the same bits."""
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


def circuit(n, max_k, seed, count=60):
    rng = np.random.default_rng(seed)
    gates = []
    for _ in range(count):
        k = int(rng.integers(1, min(max_k, n) + 1))
        g = wl.random_gate(n, k, rng)
        free = [q for q in range(n) if q not in g.targets]
        if k <= 2 and free and rng.random() < 0.25:
            c = int(rng.integers(1, len(free) + 1))
            g = wl.Gate(g.targets, g.matrix, tuple(int(q) for q in rng.choice(free, c, replace=False)), "c")
        gates.append(g)
    return gates


def run(B, n, f, psi=None, basis=None, timings=False):
    from paper_2602_09604_gb300.state import DeviceState
    st = DeviceState(n)
    if psi is not None:
        st.load(psi)
        st.apply(f, timings=timings)
    else:
        B.sv_init_apply(st.h, basis, f, timings=timings)
    B.sv_device_status()
    out = st.store()
    st.free()
    return out


# the largest error of one fused gate on a unit vector is (2^(k+1) + 2) 2^-24; a circuit adds its gates'
def bound(B, f):
    return sum((2 ** (B.sv_fused_get_info(f, i)["k"] + 1) + 2) * 2.0 ** -24 for i in range(B.sv_fused_count(f)))


@pytest.mark.parametrize("n", [3, 5, 6, 9, 11, 12, 13, 14, 17, 20, 22])
@pytest.mark.parametrize("max_k", [1, 2, 3, 4, 5])
def test_passes_match_oracle_and_single_launches(B, n, max_k):
    rng = np.random.default_rng(1000 * n + max_k)
    gates = circuit(n, max_k, seed=10 * n + max_k)
    psi = wl.random_state(n, rng).astype(np.complex64)
    f = B.sv_fuse_circuit(gates, n, max_k=max_k)
    tol = bound(B, f)
    got = run(B, n, f, psi=psi)
    again = run(B, n, f, psi=psi)
    one = run(B, n, f, psi=psi, timings=True)
    ref = psi.astype(np.complex128)
    threads = oracle.default_threads()
    for g in gates:
        oracle.apply_gate(ref, n, g, threads)
    assert np.array_equal(got.view(np.uint64), again.view(np.uint64))
    assert oracle.l2_error(ref, got) <= tol
    assert oracle.l2_error(one.astype(np.complex128), got) <= 2 * tol
    basis = int(rng.integers(0, 1 << n))
    lazy = run(B, n, f, basis=basis)
    assert oracle.l2_error(run(B, n, f, basis=basis, timings=True).astype(np.complex128), lazy) <= 2 * tol
    B.sv_fused_free(f)


@pytest.mark.parametrize("n", [11, 15, 19])
def test_tensor_core_circuits_keep_order_and_bits(B, n):
    rng = np.random.default_rng(n)
    gates = circuit(n, 3, seed=n) + wl.random_grid_circuit(wl.Grid(1, n), 6, seed=n) + circuit(n, 3, seed=n + 1)
    psi = wl.random_state(n, rng).astype(np.complex64)
    f = B.sv_fuse_circuit(gates, n, max_k=5, precision=B.PREC_BF16X3, tc_min_k=4)
    paths = {B.sv_fused_get_info(f, i)["path"] for i in range(B.sv_fused_count(f))}
    assert B.PATH_TC_BF16X3 in paths and paths - {B.PATH_TC_BF16X3}
    got, one = run(B, n, f, psi=psi), run(B, n, f, psi=psi, timings=True)
    assert np.array_equal(got.view(np.uint64), one.view(np.uint64))
    B.sv_fused_free(f)


@pytest.mark.parametrize("warm", [False, True])
def test_apply_in_a_captured_graph(B, warm):
    """Captured before any plan exists (one launch per gate) and after (passes): replays give the
    same state as an ordinary call."""
    import torch
    from paper_2602_09604_gb300.state import DeviceState
    n = 13
    gates = circuit(n, 3, seed=77)
    f = B.sv_fuse_circuit(gates, n, max_k=3)
    tol = 2 * bound(B, f)
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        st = DeviceState(n, stream=s)
        if warm:
            st.init(0)
            st.apply(f)
        s.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=s):
            st.apply(f)
        st.init(5)
        graph.replay()
        s.synchronize()
        got = st.store()
        st.init(5)
        st.apply(f, timings=True)
        want = st.store()
    assert oracle.l2_error(want.astype(np.complex128), got) <= tol
    st.free()
    B.sv_fused_free(f)
