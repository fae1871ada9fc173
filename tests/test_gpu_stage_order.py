"""Circuits with a tensor-core gate anywhere keep their order through sv_init_apply too, in the part
that runs on the small state and in the rest: calls with and without timing records (one launch per
gate, staged passes) give the same bits."""
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


def spread(n, qubits, k, count, rng):
    return [wl.random_gate(n, k, rng, targets=tuple(int(q) for q in rng.choice(qubits, k, replace=False))) for _ in range(count)]


def circuit(n, kind, rng):
    low, high = list(range(n - 4)), list(range(n - 4, n))
    wide = wl.random_gate(n, 5, rng, targets=(low[1], *high))   # names the last qubits: not in the small part
    if kind == "rest":       # tensor-core gates only after the small part
        return spread(n, low, 2, 50, rng) + [wide] + spread(n, low + high, 2, 30, rng) + spread(n, low + high, 5, 4, rng)
    if kind == "small":      # and only in it
        cover = [wl.random_gate(n, 2, rng, targets=(high[0], high[1])), wl.random_gate(n, 2, rng, targets=(high[2], high[3]))]
        return spread(n, low, 2, 30, rng) + spread(n, low, 5, 4, rng) + cover + spread(n, low + high, 2, 50, rng)
    near = low[:9]           # in it, on a small state that is too small for the tensor cores
    return spread(n, near, 5, 6, rng) + [wl.random_gate(n, 2, rng, targets=(near[0], n - 1))] + spread(n, low + high, 2, 50, rng)


@pytest.mark.parametrize("kind", ["rest", "small", "near"])
@pytest.mark.parametrize("n", [14, 20])
def test_lazy_starts_keep_order_and_bits(B, n, kind):
    from paper_2602_09604_gb300.state import DeviceState
    rng = np.random.default_rng(n)
    gates = circuit(n, kind, rng)
    f = B.sv_fuse_circuit(gates, n, mode=B.FUSE_NONE, precision=B.PREC_BF16X3, tc_min_k=4, start_qubits=9 if kind == "near" else 0)
    st = DeviceState(n)
    rec = B.sv_init_apply(st.h, 3, f, timings=True)
    want = st.store()
    assert 0 < sum(r["path"] == B.PATH_AUTO for r in rec) < len(rec)
    B.sv_init_apply(st.h, 3, f)
    got = st.store()
    assert np.array_equal(got.view(np.uint64), want.view(np.uint64))
    assert oracle.l2_error(oracle.run_circuit(n, gates, 3, threads=oracle.default_threads()), got) <= 1e-4
    B.sv_fused_free(f)
    st.free()


@pytest.mark.parametrize("n,m,max_k", [(20, 14, 3), (26, 24, 6), (27, 26, 5)])
def test_light_cones_without_timing_records(B, n, m, max_k):
    from paper_2602_09604_gb300.state import DeviceState
    rng = np.random.default_rng(7 * n + m)
    gates = []
    for _ in range(120):
        k = int(rng.integers(1, 3))
        nc = int(rng.integers(0, 3)) if rng.random() < 0.2 else 0
        qs = [int(q) for q in rng.permutation(n)]
        gates.append(wl.Gate(tuple(qs[:k]), wl.random_unitary(1 << k, rng), tuple(qs[k:k + nc])))
    f = B.sv_fuse_circuit(gates, n, max_k=max_k, precision=B.PREC_BF16X3, tc_min_k=4, start_qubits=m)
    tc = any(B.sv_fused_get_info(f, i)["path"] == B.PATH_TC_BF16X3 for i in range(B.sv_fused_count(f)))
    st = DeviceState(n)
    B.sv_init_apply(st.h, 9, f, timings=True)
    want = st.buf.clone()
    B.sv_init_apply(st.h, 9, f)
    if tc:
        assert bool((st.buf == want).all())
    else:
        assert float((st.buf.double() - want.double()).norm()) <= 1e-4
    B.sv_fused_free(f)
    st.free()
