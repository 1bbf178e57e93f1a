"""Accuracy of the FP32 row phase on column-major fields: J of a given curve against
FP64, beside the row-major row phase's (the dense form) on the same curves.  Both carry
the roundings of one transform pair, so the rms error over sixteen curves is held to
1.2 times the row-major one's (the spread of an rms over sixteen) plus half a rounding."""
import numpy as np
import pytest
import torch

from paper_2301_11704_gb300 import gen
from paper_2301_11704_gb300.curve import KSCurve

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,Ns", [(32, 1000), (64, 1000), (64, 6000), (128, 1000), (128, 4096), (256, 1000), (256, 4096)])
def test_cost_error_of_the_fp32_row_phase(N, Ns):
    sp = gen.workload({32: 0, 64: 1, 128: 2, 256: 4}[N])[0]
    up, um = gen.end_points(sp)
    S = gen.mapping_scale(Ns)
    err = {"auto": [], "dense": []}
    for seed in range(16):
        ref = KSCurve(sp.L, N, Ns, S, up, um, precision="fp64")
        rng = np.random.default_rng(seed)
        ref.init_trial(0.0, None, rng.uniform(0.05, 0.2, 4), gen.perturbation_fields(N, sp.L, seed + 1, 4))
        u = ref.get_state().float()
        ref.set_state(u.double())
        J = np.sqrt(ref.cost()[0])
        ref.close()
        for form in err:
            c = KSCurve(sp.L, N, Ns, S, up, um, precision="fp32", s_transform=form)
            c.set_state(u)
            err[form].append(np.sqrt(c.cost()[0]) / J - 1)
            c.close()
    a, d = (float(np.sqrt(np.mean(np.square(err[f])))) for f in ("auto", "dense"))
    print("J error N=%d Ns=%d: column form %.2e, row-major %.2e" % (N, Ns, a, d))
    assert a <= 1.2 * d + 3e-8
