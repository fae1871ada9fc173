"""Every form of the staged-pass kernel (many small CTAs or few large ones, each largest gate size) on a
circuit whose plan takes it, against the oracle."""
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


@pytest.mark.parametrize("n", [13, 20, 22, 23])
@pytest.mark.parametrize("kmax", [1, 2, 3, 4, 5])
def test_form(B, n, kmax):
    import torch
    from paper_2602_09604_gb300.state import DeviceState
    rng = np.random.default_rng(10 * n + kmax)
    # layers of kmax-qubit gates that share one tile, high and low targets
    gates = []
    for _ in range(3):
        pool = [int(q) for q in rng.permutation(9)] + [int(q) for q in rng.choice(np.arange(9, n), 2, replace=False)]
        for i in range(0, len(pool) - kmax + 1, kmax):
            gates.append(wl.random_gate(n, kmax, rng, targets=tuple(pool[i:i + kmax])))
        if kmax >= 3:   # unfused, a dense gate of three qubits
            gates.append(wl.Gate((pool[0],), wl.random_unitary(2, rng), (pool[1], n - 1)))
    f = B.sv_fuse_circuit(gates, n, mode=B.FUSE_NONE)
    sizes = [B.sv_fused_get_info(f, i)["k"] for i in range(B.sv_fused_count(f))]
    passes = [s for s in B.sv_fused_plan_passes(f) if s["tile"]]
    assert any(max(sizes[g] for g in s["gates"]) == kmax for s in passes)
    many = (1 << (n - bin(passes[0]["tile"]).count("1"))) >= 2 * torch.cuda.get_device_properties(0).multi_processor_count
    assert many == (n >= 22)
    psi = wl.random_state(n, rng).astype(np.complex64)
    st = DeviceState(n)
    for _ in range(8):   # the first calls of a short circuit go gate by gate
        st.load(psi)
        st.apply(f)
    got = st.store()
    ref = psi.astype(np.complex128)
    for g in gates:
        oracle.apply_gate(ref, n, g, oracle.default_threads())
    # one fused gate's error on a unit vector is at most (2^(k+1) + 2) 2^-24
    assert oracle.l2_error(ref, got) <= sum((2 ** (k + 1) + 2) * 2.0 ** -24 for k in sizes)
    B.sv_fused_free(f)
    st.free()
