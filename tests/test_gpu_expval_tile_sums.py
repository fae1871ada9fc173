"""Pauli strings on the sizes that take tile passes (26 qubits and more), every string against 64-bit
sums: more strings on one x mask than a run holds, several passes filled to their limits, masks that use
up a tile's qubits, z on every index bit; a state without structure to the size of its random
rounding, a state that repeats one pattern to the bound."""
import numpy as np
import pytest

from paper_2602_09604_gb300 import build as libbuild

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    libbuild.build()
    import torch
    assert torch.cuda.is_available()
    from paper_2602_09604_gb300 import binding
    return binding


def strings(n, rng):
    out = []
    for q in range(n - 1):                                        # chains: four masks of two, z pairs
        out += [(3 << q, 0), (3 << q, 3 << q), (3 << q, 1 << q), (0, 3 << q)]
    out += [(0, 1 << q) for q in range(n)] + [(1 << q, 1 << q) for q in range(0, n, 3)]
    out += [(0, int(rng.integers(0, 1 << n))) for _ in range(6)]
    one = 1 << 9 | 1 << 3                                         # 41 strings of one mask: cut into two runs
    out += [(one, int(rng.integers(0, 1 << n))) for _ in range(41)]
    full = sum(1 << q for q in (6, 9, 13, 17, 20, 23, n - 1))     # with qubits 0-4 the whole of a tile
    out += [(full, 0), (full | 21, full), (full | 10, int(rng.integers(0, 1 << n)))]
    out += [((1 << n) - 1, 0)]                                    # fits no tile
    return out


def gauss(n, torch):
    gen = torch.Generator(device="cuda").manual_seed(n)
    return torch.randn(1 << n, 2, device="cuda", generator=gen)


def pattern(n, torch):
    """The same eight amplitudes on the qubits that a thread's sums run over, whatever the others hold."""
    gen = torch.Generator(device="cuda").manual_seed(n)
    eight = torch.randn(8, 2, device="cuda", generator=gen)
    return eight[(torch.arange(1 << n, device="cuda") >> 7) & 7]


@pytest.mark.parametrize("n,make", [(26, gauss), (27, gauss), (26, pattern)])
def test_against_64_bits(B, n, make):
    import torch
    from paper_2602_09604_gb300.state import DeviceState
    rng = np.random.default_rng(n)
    amps = make(n, torch)
    amps = (amps / torch.linalg.vector_norm(amps.double())).float().contiguous()
    st = DeviceState(n)
    B.sv_load(st.h, amps.data_ptr(), False)
    todo = strings(n, rng)
    order = rng.permutation(len(todo))
    todo = [todo[i] for i in order]
    got = B.sv_expval_pauli(st.h, [x for x, _ in todo], [z for _, z in todo])
    assert np.array_equal(got, B.sv_expval_pauli(st.h, [x for x, _ in todo], [z for _, z in todo]))
    alone = np.array([B.sv_expval_pauli(st.h, [x], [z])[0] for x, z in todo[::9]])
    assert (alone != got[::9]).any()   # the other kernel's sums: tile passes did run
    st.free()
    del st
    psi = torch.view_as_complex(amps).to(torch.complex128)
    index = torch.arange(1 << n, device="cuda")
    eps = 2.0 ** -24
    for x in sorted({x for x, _ in todo}):
        partner = psi[index ^ x]
        size = (partner.abs() * psi.abs())
        # A term has two roundings and takes part in three of sums, each of them at most eps of a value that
        # is at most the sum of its terms' sizes.  The bound is 5 eps of all sizes (and its square).  Where
        # they are independent (uniform, deviation eps / sqrt 3) their variance is at most
        # eps^2 / 3 (2 + 2 + 4 + 8) sum size^2, twice that for x != 0, where a term stands for two.
        bound = 5.01 * eps * float(size.sum())
        sigma = eps * (16 / 3 * (2 if x else 1) * float((size * size).sum())) ** 0.5
        tol = bound if make is pattern else 6 * sigma
        if x == (1 << n) - 1:   # the one-mask kernel: 15 serial sums a term
            tol = 17.1 * eps * float(size.sum())
        del size
        p = partner.conj_physical_() * psi
        del partner
        for i, (xi, z) in enumerate(todo):
            if xi != x:
                continue
            sign = torch.ones(1, dtype=torch.float64, device="cuda")
            for q in range(n):
                sign = torch.cat((sign, -sign if (z >> q) & 1 else sign))
            c = bin(x & z).count("1") & 3
            want = float((p.real * sign).sum()) * (1, 0, -1, 0)[c] + float((p.imag * sign).sum()) * (0, -1, 0, 1)[c]
            assert abs(got[i] - want) <= tol, (x, z, got[i] - want, tol)
