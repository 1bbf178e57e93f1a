"""Batches in the forms that s_transform names, their launch-shape choices and the
order of their reads: "fft" runs the one-CTA FFT form and, from F = 1024 on, the
one-CTA-per-mode four-step form, each curve against its own single-curve run; the
autotuner tries a knob only where a curve of the batch runs the kernels it shapes."""
import numpy as np
import pytest
import torch

from paper_2301_11704_gb300 import gen
from paper_2301_11704_gb300.batch import KSBatch
from tests.test_gpu_batch import _four_step_specs, _inputs

pytestmark = pytest.mark.gpu


def _batch(specs, **kw):
    ins = [_inputs(s) for s in specs]
    b = KSBatch(specs, [i[0] for i in ins], [i[1] for i in ins], conv="jarc", **kw)
    b.init_trial(np.array([i[2] for i in ins]), [i[3] for i in ins])
    return b, ins


def test_get_state_returns_a_finished_copy():
    """The tensor may go to any stream or thread: nothing of the batch's stream is
    pending when get_state returns, here behind descent steps of several milliseconds."""
    b, _ = _batch(_four_step_specs([(64, 1500), (128, 2100)]), precision="fp64")
    b.descend(1)
    b.descend_async(100)
    b.get_state(0)
    assert b.stream.query()
    b.close()
