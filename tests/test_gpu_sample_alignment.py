"""sv_sample_noalloc on states that lie at any float boundary: the same samples as from an aligned
state (the same sums in the same order), and an error for an address between floats."""
import numpy as np
import pytest

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


@pytest.mark.parametrize("n", [2, 5, 9, 14, 15, 18])
def test_offset_states_give_the_same_samples(B, n):
    import torch
    from paper_2602_09604_gb300.state import DeviceState
    rng = np.random.default_rng(n)
    st = DeviceState(n)
    st.load(wl.random_state(n, rng))
    u = np.concatenate((rng.random(200), [0.0, np.nextafter(1.0, 0.0)]))
    want = st.sample(u)
    wide = torch.empty(st.buf.numel() + 8, dtype=torch.float32, device="cuda")
    for off in range(6):
        wide[off:off + st.buf.numel()] = st.buf
        got = B.sv_sample_noalloc(wide.data_ptr() + 4 * off, n, st.stream.cuda_stream, u)
        assert np.array_equal(got, want), off
    with pytest.raises(B.SvError) as e:
        B.sv_sample_noalloc(wide.data_ptr() + 2, n, st.stream.cuda_stream, u)
    assert e.value.code == B.SV_EINVAL
    assert B.sv_sample_noalloc(wide.data_ptr() + 2, n, st.stream.cuda_stream, []).size == 0
    st.free()
