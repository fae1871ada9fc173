"""Pauli strings that share a read pass through shared-memory tiles (many x masks, or more z masks
than one pass of the one-mask kernel takes) against the oracle, around the tile size (2^12
amplitudes) and with masks inside, across and outside a tile; and the same strings one at a time,
which run on the one-mask kernel."""
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


def chain(n):
    out = []
    for q in range(n - 1):
        out += [{q: p, q + 1: p} for p in "XYZ"] + [{q: "X", q + 1: "Y"}]
    out += [{q: p} for q in range(n) for p in "XYZ"]
    out += [{0: "X", n - 1: "Y", n // 2: "Z"}, {q: "X" for q in range(n)}, {q: "Y" for q in range(0, n, 2)}, {}]
    return out


@pytest.mark.parametrize("n", [11, 12, 13, 18])
def test_chain_terms_match_oracle(B, n):
    from paper_2602_09604_gb300.state import DeviceState
    psi = wl.random_state(n, np.random.default_rng(n))
    st = DeviceState(n)
    st.load(psi)
    strings = chain(n)
    got = st.expval(strings)
    assert np.array_equal(got, st.expval(strings))
    # fp32 terms (relative error 2^-23 each) and fp32 sums of at most 16 of them, then wider sums:
    # at most 20 * 2^-24 of the sum of |terms| <= 1
    ref, threads = psi.astype(np.complex64).astype(np.complex128), oracle.default_threads()
    for t, g in zip(strings, got):
        assert abs(g - oracle.expval_pauli(ref, n, t, threads).real) <= 20 * 2.0 ** -24, (n, t)
    one = np.array([st.expval([t])[0] for t in strings])
    assert np.max(np.abs(one - got)) <= 40 * 2.0 ** -24
    st.free()


def test_tiles_match_one_string_at_a_time(B):
    """26 qubits, the smallest state whose strings share tile passes."""
    import torch
    from paper_2602_09604_gb300.state import DeviceState
    n = 26
    gen = torch.Generator(device="cuda").manual_seed(3)
    psi = torch.randn(1 << n, 2, device="cuda", generator=gen)
    psi = (psi / torch.linalg.vector_norm(psi.double())).float().contiguous()
    st = DeviceState(n)
    B.sv_load(st.h, psi.data_ptr(), False)
    strings = chain(n)
    got = st.expval(strings)
    assert np.array_equal(got, st.expval(strings))
    one = np.array([st.expval([t])[0] for t in strings])
    assert np.max(np.abs(one - got)) <= 40 * 2.0 ** -24
    amps = torch.view_as_complex(psi).to(torch.complex128)
    probs = amps.abs().square().view(-1, 4096)
    sign = torch.tensor([(-1.0) ** bin(i & 3).count("1") for i in range(4096)], dtype=torch.float64, device="cuda")
    assert abs(got[strings.index({0: "Z", 1: "Z"})] - float((probs * sign).sum())) <= 20 * 2.0 ** -24
    st.free()
