"""Batches in the forms that s_transform names, their launch-shape choices and the
order of their reads: "fft" runs the one-CTA FFT form and, from F = 1024 on, the
one-CTA-per-mode four-step form, each curve against its own single-curve run; the
autotuner tries a knob only where a curve of the batch runs the kernels it shapes."""
import numpy as np
import pytest

import oracle
from paper_2301_11704_gb300.batch import KSBatch
from paper_2301_11704_gb300.curve import KSCurve
from tests.test_gpu_batch import _four_step_specs, _inputs
from tests.test_gpu_parity import rel_2

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


# Between s-forms: 1e-10 in FP64 as in test_gpu_fft4.py, 2e-5 in FP32 as in test_gpu_batch.py
# (a hundred steps or fewer); 1e-10 against the oracle.
FFT_TOL = dict(fp64=1e-10, fp32=2e-5)


@pytest.mark.parametrize("precision,sizes,kw", [
    ("fp64", [(32, 130), (64, 300), (32, 700), (64, 1100), (128, 2000)], {}),            # F 512 (one-CTA) to 4096
    ("fp32", [(32, 130), (64, 300), (32, 700), (64, 1500), (128, 2100), (32, 4096)], {}),   # and 8192
    ("fp64", [(32, 200), (32, 400), (64, 700)], dict(adjoint="discrete")),
    ("fp64", [(32, 300), (64, 600)], dict(symmetry=5)),
    ("fp32", [(32, 300), (64, 1500)], dict(symmetry=5)),
    ("fp64", [(32, 65), (32, 400), (64, 1100)], dict(scheme="implicit", dtau=0.2)),
    ("fp32", [(32, 65), (32, 400), (64, 1100)], dict(scheme="implicit", dtau=0.2)),
])
def test_fft_batch_matches_independent_curves(precision, sizes, kw):
    """Before and after the autotuner, which tries every split of every length."""
    specs = _four_step_specs(sizes)
    b, ins = _batch(specs, precision=precision, s_transform="fft", **kw)
    splits = b.tuning()["splits"]
    assert splits and all(f1 * f2 == F >= 1024 for F, (f1, f2) in splits.items())
    curves = []
    for s, (up, um, amps, vp) in zip(specs, ins):
        c = KSCurve(s.L, s.N, s.Ns, s.S, up, um, precision=precision, s_transform="dense", **dict(dict(dtau=s.dtau), **kw))
        c.init_trial(0.0, None, amps, vp)
        curves.append(c)
    tol, done = FFT_TOL[precision], np.zeros(len(specs), dtype=int)
    for tuned in (False, True):
        if tuned:
            assert set(b.autotune(2)["splits"]) == set(splits)
        out = b.descend(10)
        steps = np.array([x["step"] for x in b.scalars()])
        for k, c in enumerate(curves):
            ref = c.descend(int(steps[k] - done[k]))
            x, xc = b.get_state(k).double().cpu().numpy(), c.get_state().double().cpu().numpy()
            assert rel_2(x, xc) <= tol, (k, specs[k], tuned)
            assert abs(out["J"][k] - ref["J"]) <= tol * ref["J"]
        done = steps
    b.close()


def test_fft_batch_matches_the_oracle_fp64():
    specs = _four_step_specs([(32, 700), (64, 1200), (32, 300), (64, 500)])
    b, ins = _batch(specs, precision="fp64", s_transform="fft")
    out = b.descend(10)
    for k, (s, (up, um, amps, vp)) in enumerate(zip(specs, ins)):
        U = oracle.curve_init(s.M, s.S, up, um, amps=amps, vp=vp)
        Uo, _, sco, _ = oracle.curve_descend(U, s.L, s.S, 10, dtau=s.dtau)
        xo = oracle.curve_physical(Uo)
        assert np.abs(b.get_state(k).cpu().numpy() - xo).max() <= 1e-10 * np.abs(xo).max()
        assert abs(out["J_arc"][k] - sco["J_arc"]) <= 1e-10 * sco["J_arc"]
    b.close()


@pytest.mark.parametrize("adjoint", ["paper", "discrete"])
def test_clustered_step_fp64_matches_the_dense_form(adjoint):
    """N = 16, N_s = 1000 in FP64: the clustered four-step form's one-launch step."""
    s = _four_step_specs([(32, 1000)])[0]
    N, L = 16, 22.0
    up, um = np.zeros(N), np.zeros(N)
    amps, vp = np.full(2, 0.1), np.stack([np.sin(2 * np.pi * q * np.arange(N) / N) for q in (1, 2)])
    res = []
    for form in ("fft4c", "dense"):
        c = KSCurve(L, N, s.Ns, s.S, up, um, dtau=1e-3, precision="fp64", adjoint=adjoint, s_transform=form)
        c.init_trial(0.0, None, amps, vp)
        out = c.descend(20)
        res.append((out["J"], c.get_state().cpu().numpy()))
        c.close()
    (Ja, xa), (Jb, xb) = res
    assert abs(Ja - Jb) <= 1e-10 * Jb and np.abs(xa - xb).max() <= 1e-10 * np.abs(xb).max()
