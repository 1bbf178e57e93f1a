"""The bounded wait of the column form for a step's decision: a wait that runs out (its
bound set to give up at once) is reported as KS_ETIMEOUT and leaves a usable context."""
import pytest
import torch

from paper_2301_11704_gb300 import _native
from tests.test_gpu_failure import _curve as _trial

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,N,Ns,steps", [
    ("fp32", 64, 200, 1),      # a CTA per column (L = 256)
    ("fp32", 64, 9000, 20),    # 32 values per thread, graph replay
    ("fp64", 128, 300, 20),    # a CTA per column, FP64
    ("fp64", 64, 600, 1),      # two CTAs per column
    ("fp64", 32, 1100, 20),    # four
])
def test_expired_wait_for_the_decision(precision, N, Ns, steps):
    """A step whose decision is not taken in time is not applied: KS_ETIMEOUT, also from
    every later read, until the curve is re-initialised; then as a fresh curve."""
    c, (amps, vp) = _trial(N, Ns, precision)
    ref, _ = _trial(N, Ns, precision)
    J2_ref, out_ref = ref.cost()[0], ref.descend(steps)
    u_ref = ref.get_state()
    ref.close()
    u0 = c.get_state()
    c.debug_wait_limit(-1)
    with pytest.raises(_native.KSError) as err:
        c.descend(steps)
    assert err.value.status == _native.KS_ETIMEOUT
    with pytest.raises(_native.KSError):
        c.scalars()
    assert torch.equal(c.get_state(), u0)
    c.init_trial(0.0, None, amps, vp)
    assert c.cost()[0] == J2_ref
    out = c.descend(steps)
    assert out["J"] == out_ref["J"] and torch.equal(c.get_state(), u_ref)
    c.close()
