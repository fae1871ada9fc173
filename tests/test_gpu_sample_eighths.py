"""Targets just below the end of an eighth of a chunk: its sum decides whether the walk starts there
or behind it, so it has to be as exact as fp64 sums are.  States of one repeated amplitude, whose
rounding adds up alike in every thread; one chunk, so that the target is u times the norm that the
same call returns; the answer by exact rational arithmetic."""
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


# 2^-47 and 2^66: amplitudes whose squares fp32 cannot split exactly, or not add
@pytest.mark.parametrize("scale", [1.0, 2.0 ** -47, 2.0 ** 66])
def test_targets_at_the_ends_of_eighths(B, scale):
    from paper_2602_09604_gb300.state import DeviceState
    n, eighth = 14, 1 << 11
    st = DeviceState(n)
    for amp in np.float32(scale) * np.random.default_rng(14).uniform(0.002, 0.02, 24).astype(np.float32):
        c = np.complex64(amp * (1 + 0.75j))
        st.load(np.full(1 << n, c, dtype=np.complex64))
        p = Fraction(float(c.real)) ** 2 + Fraction(float(c.imag)) ** 2
        _, norm = B.sv_sample_norm(st.h, [])
        us, want = [], []
        for e in range(1, 8):
            # fp64 sums of 64 squares a chain and a few adds are within 2^-47 of the exact ones; the
            # target lies 2^-46 below the end
            u = float(e * eighth * p * (1 - Fraction(1, 1 << 46)) / Fraction(norm))
            target = Fraction(u * norm)
            us.append(u)
            want.append(int(target / p))   # p (i + 1) > target first at i = floor(target / p)
        assert want == [e * eighth - 1 for e in range(1, 8)]
        assert st.sample(np.array(us)).tolist() == want, amp
    st.free()
