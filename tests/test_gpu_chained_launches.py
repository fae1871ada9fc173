"""Gate kernels one behind the other at the sizes where two of them share the GPU: chaining them must not
make a gate slower than the same gates on a state half as large by more than the size itself
explains (these kernels are bound by latency there), and the states stay right."""
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


def alternating(n, a, b, rng):
    """Gates that share a qubit and fit no common tile: each has its own launch."""
    k = len(a)
    return [wl.random_gate(n, k, rng, targets=t) for _ in range(6) for t in (a, b)]


CASES = {
    "five_high": ((5, 6, 7, 8, 9), (9, 10, 11, 12, 13)),
    "five_mixed": ((0, 5, 6, 7, 8), (0, 9, 10, 11, 12)),
    "six_mixed": ((0, 1, 2, 5, 6, 7), (1, 3, 4, 8, 9, 10)),
}


@pytest.mark.parametrize("name", list(CASES))
def test_nineteen_qubits_take_little_more_than_eighteen(B, name):
    import torch
    from paper_2602_09604_gb300.state import DeviceState
    times = {}
    for n in (18, 19):
        rng = np.random.default_rng(n)
        gates = alternating(n, *CASES[name], rng)
        f = B.sv_fuse_circuit(gates, n, mode=B.FUSE_NONE)
        assert all(len(s["gates"]) == 1 for s in B.sv_fused_plan_passes(f))
        st = DeviceState(n)
        st.init(0)
        st.apply(f)
        got = st.store()
        tol = sum((2 ** (len(g.targets) + 1) + 2) * 2.0 ** -24 for g in gates)
        assert oracle.l2_error(oracle.run_circuit(n, gates, 0, threads=oracle.default_threads()), got) <= tol
        runs = []
        for _ in range(15):
            begin, end = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            torch.cuda.synchronize()
            begin.record(st.stream)
            for _ in range(20):
                st.apply(f)
            end.record(st.stream)
            torch.cuda.synchronize()
            runs.append(begin.elapsed_time(end))
        times[n] = sorted(runs)[7]
        B.sv_fused_free(f)
        st.free()
    # measured 1.1 and less; 1.37 to 1.5 where the second kernel's CTAs crowded beside the first one's
    assert times[19] <= 1.25 * times[18], times


@pytest.mark.parametrize("n", [18, 19, 20, 21, 22])
@pytest.mark.parametrize("k", [1, 2, 3, 4, 5, 6])
def test_launch_forms_match_the_oracle(B, n, k):
    """Chains of every gate size around the sizes where the launch form changes."""
    from paper_2602_09604_gb300.state import DeviceState
    rng = np.random.default_rng(n * k)
    gates = []
    for i in range(12):
        p = [int(q) for q in rng.permutation(n)]
        c = tuple(p[k:k + 7 - k]) if k <= 3 and i % 3 == 0 else ()
        gates.append(wl.Gate(tuple(p[:k]), wl.random_unitary(1 << k, rng), c, "g"))
    f = B.sv_fuse_circuit(gates, n, max_k=k)
    st = DeviceState(n)
    for _ in range(3):
        st.init(1)
        st.apply(f)
    tol = sum((2 ** (B.sv_fused_get_info(f, i)["k"] + 1) + 2) * 2.0 ** -24 for i in range(B.sv_fused_count(f)))
    assert oracle.l2_error(oracle.run_circuit(n, gates, 1, threads=oracle.default_threads()), st.store()) <= tol
    B.sv_fused_free(f)
    st.free()
