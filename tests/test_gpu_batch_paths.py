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


def test_autotune_leaves_the_dense_tile_without_dense_curves():
    """Column-form curves have no s-phase tile: the row phase's two widths (2 + 3 steps
    each) are all that is timed, on the callers' curves."""
    b, _ = _batch(_four_step_specs([(64, 300), (128, 400)]), precision="fp32")
    tune = b.autotune(3)
    assert tune["dense_tile"] == 0
    assert [x["step"] for x in b.scalars()] == [10, 10]
    b.close()


def test_autotune_tries_the_dense_tile_of_dense_curves():
    """One dense curve (N_s = 40) of 64 columns beside a column-form one: both widths are timed."""
    b, _ = _batch(_four_step_specs([(64, 40), (64, 300)]), precision="fp32", s_transform="dense")
    tune = b.autotune(3)
    assert tune["dense_tile"] in (32, 64)
    assert [x["step"] for x in b.scalars()] == [20, 20]
    b.close()


@pytest.mark.parametrize("form,precision,sections", [("auto", "fp32", 16), ("auto", "fp64", 8), ("dense", "fp32", 8),
                                                     ("fft", "fp32", 8), ("dense", "fp64", 8)])
def test_row_sections_of_a_new_batch(form, precision, sections):
    """16 sections per row CTA only where FP32 curves run the column form."""
    b, _ = _batch(_four_step_specs([(64, 300), (128, 400)]), precision=precision, s_transform=form)
    assert b.tuning()["row_sections"] == sections
    b.close()
