"""Limits of the column form: its bounded wait for a step's decision (a wait that runs
out, its bound set to give up at once, is reported as KS_ETIMEOUT and leaves a usable
context), and the range of |G| in FP32 storage: amplitudes where every coefficient of G
is an FP32 number but w_m g^2 is not.  |G| is compared with the FP64 quadrature of the
curve's own G, which comes back through one FP32 transform: some ten roundings, 2e-5 at
most."""
import numpy as np
import pytest
import torch

from paper_2301_11704_gb300 import _native
from paper_2301_11704_gb300.curve import KSCurve
from tests.test_gpu_failure import _curve as _trial
from tests.test_gpu_fft4 import _curve

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


# the plans of 8, 16 and 32 values per thread; weights from 6e-7 to 8e5
@pytest.mark.parametrize("N,Ns", [(64, 700), (32, 3000), (32, 5000)])
@pytest.mark.parametrize("S,gmax", [(None, 1e18), (1e-3, 3e-19)])
def test_gradient_norm_keeps_the_range_of_fp32(N, Ns, S, gmax):
    L = 22.0 * N / 64
    X = _curve(N, Ns, L, N + Ns)
    S = 0.1 * (Ns - 1) if S is None else S

    def make(scale):
        u = torch.from_numpy(scale * X).float()
        c = KSCurve(L, N, Ns, S, u[0].double().numpy(), u[-1].double().numpy(), u_init=u, precision="fp32", dtau=1e-3)
        return c, c.gradient()[0].double().cpu().numpy()
    # the scale at which the largest coefficient of G is gmax (G is cubic for large curves, linear for small)
    scale, power = (1e5, 1.0 / 3.0) if gmax > 1 else (1e-20, 1.0)
    for _ in range(2):
        c, g = make(scale)
        scale *= (gmax * N / np.abs(np.fft.rfft(g, axis=1)).max()) ** power
        c.close()
    c, g = make(scale)
    th = np.arange(Ns)[1:-1] * np.pi / (Ns - 1)
    want = np.sqrt((np.pi / (Ns - 1) * S / np.sin(th) ** 2 * (L / N) * (g[1:-1] ** 2).sum(1)).sum())
    assert abs(c.scalars()["G_norm"] - want) <= 2e-5 * want
    c.descend_async(1)   # the deferred sum of a descent step, of the same G
    assert abs(c.scalars()["G_norm"] - want) <= 2e-5 * want
    c.close()
