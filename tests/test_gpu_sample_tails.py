"""Samples whose probability is tiny against the amplitudes after them: the smallest index whose
cumulative probability exceeds u times the total, by exact rational arithmetic, where a few
amplitudes of 1e-12 lie before amplitudes of order one (targets lie halfway into an outcome's share,
far from rounding).  At each level: in a thread, across threads, warps, steps, eighths and chunks."""
from fractions import Fraction

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


@pytest.mark.parametrize("span", [1, 8, 256, 2048, 1 << 14])
@pytest.mark.parametrize("n", [5, 9, 12, 14, 16, 18, 20])
def test_small_probabilities_before_large_ones(B, n, span):
    from paper_2602_09604_gb300.state import DeviceState
    N = 1 << n
    if N < 4 * span:
        pytest.skip("state of fewer than four such spans")
    rng = np.random.default_rng(n * span)
    st = DeviceState(n)
    for _ in range(12):
        # small amplitudes in the spans up to the first large one's, and in that span before it
        first = int(rng.integers(1, N // span))
        slots = np.arange(max(0, first - 5), first + 1)
        small = sorted(set(int(rng.integers(s * span, (s + 1) * span)) for s in slots))
        at = max(small[-1] + 1, int(rng.integers(first * span, (first + 1) * span)))
        large = [i for i in (at, at + 1, at + 5 * span) if i < N]
        if not large:
            continue
        psi = np.zeros(N, dtype=np.complex64)
        psi[small] = rng.uniform(1e-12, 3e-12, len(small))
        psi[large] = rng.uniform(0.5, 1.0, len(large))
        idx = small + large
        p = [Fraction(float(psi[i].real)) ** 2 for i in idx]
        total, before, us = sum(p), Fraction(0), [0.0]
        for q in p:
            us.append(float((before + q / 2) / total))
            before += q
        st.load(psi)
        want = [idx[0]] + idx
        assert st.sample(np.array(us)).tolist() == want
        assert B.sv_sample_noalloc(st.buf.data_ptr(), n, st.stream.cuda_stream, us).tolist() == want
    st.free()
