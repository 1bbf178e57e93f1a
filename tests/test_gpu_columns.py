"""The column form of the s-contraction (one real column per CTA, right-angle
convolution of the sections' differences, column-major fields), which `auto` runs
from N_s = 64 up to 16384 (FP32) and 8192 (FP64), against the dense contraction on the
same inputs: every transform length it is built for at the edges of its range,
both adjoints, the symmetric subspaces in both storages, the descent with lambda
free, the stop at a tolerance and the asynchronous call's scalars.

FP64 agrees with the dense form to 1e-10 relative, as the other forms do.  In FP32
every result is at most 1.5 times as far from the FP64 dense form's as the FP32 dense
form's own (same arithmetic, fewer roundings) or within 2e-6, thirty roundings."""
import numpy as np
import pytest
import torch

from paper_2301_11704_gb300.curve import KSCurve
from tests.test_gpu_fft4 import _curve
from tests.test_gpu_parity import rel_2

pytestmark = pytest.mark.gpu



def _curves(N, Ns, precision, **kw):
    """The same curve in the column form, in the dense form, and dense in FP64."""
    L = 22.0 * N / 64   # the workloads' resolution: top wavenumber 9.1
    X = _curve(N, Ns, L, N + Ns, fp32=precision == "fp32")
    if kw.get("symmetry", 0):   # odd sections
        X = 0.5 * (X - np.roll(X[:, ::-1], 1, axis=1))
        if precision == "fp32":
            X = X.astype(np.float32).astype(np.float64)
    u = torch.from_numpy(X)
    S = 0.1 * (Ns - 1)

    def make(p, form):
        return KSCurve(L, N, Ns, S, X[0], X[-1], u_init=u.to(torch.float32 if p == "fp32" else torch.float64),
                       precision=p, dtau=1e-3, s_transform=form, **kw)
    return make(precision, "auto"), make(precision, "dense"), make("fp64", "dense")


def _results(c, steps):
    """Name -> value of what the curve computes; the gradient in the norm the descent applies it in."""
    J2, Ja = c.cost()
    k = 2 * np.pi * np.arange(c.nx // 2) / c.L
    pw = 0.01 / (1.0 + 0.01 * (k ** 4 - k ** 2) ** 2)
    g = np.fft.rfft(c.gradient()[0].double().cpu().numpy(), axis=1)[:, :c.nx // 2] * pw
    out = dict(J2=J2, J_arc=Ja, r=c.residual().double().cpu().numpy(), g=g)
    o = c.descend(steps)
    lam, tau = c.get_lambda_tau()
    assert o["steps"] == steps and abs(tau - steps * 1e-3) < 1e-12
    return dict(out, J=o["J"], u=c.get_state().double().cpu().numpy(), lam=lam)


def _compare(curves, precision, steps=5):
    a, b, ref = (_results(c, steps) for c in curves)
    for k in ref:
        ea, eb = rel_2(a[k], ref[k]), rel_2(b[k], ref[k])
        assert ea <= (1e-10 if precision == "fp64" else 1.5 * eb + 2e-6), (k, ea, eb)
    for c in curves:
        c.close()


# N_s at both ends of every length from 128 (the shortest) to 16384; in FP64 also every
# split of a column over a cluster (2 or 4 CTAs, classes of 256 to 4096 frequencies)
@pytest.mark.parametrize("precision,N,Ns", [
    ("fp32", 8, 64), ("fp32", 16, 127), ("fp32", 32, 128), ("fp32", 64, 129), ("fp32", 128, 256), ("fp32", 256, 257),
    ("fp32", 64, 512), ("fp32", 32, 513), ("fp32", 64, 1025), ("fp32", 16, 2048), ("fp32", 128, 2049),
    ("fp32", 8, 4097), ("fp32", 16, 8192), ("fp32", 8, 8193), ("fp32", 16, 16384),
    ("fp64", 8, 64), ("fp64", 16, 128), ("fp64", 32, 129), ("fp64", 64, 257), ("fp64", 128, 512), ("fp64", 256, 513),
    ("fp64", 32, 1024), ("fp64", 64, 1025), ("fp64", 16, 2049), ("fp64", 128, 2049), ("fp64", 8, 4097), ("fp64", 64, 4097),
    ("fp64", 8, 8192)])
def test_column_form_matches_dense(precision, N, Ns):
    _compare(_curves(N, Ns, precision), precision)


# the sections at which single FP32 curves change the row phase's values per thread
@pytest.mark.parametrize("N,Ns", [(32, 4866), (32, 4867), (32, 9735), (64, 2432), (64, 2433), (64, 4866), (64, 4867),
                                  (128, 2432), (128, 2433), (256, 2432), (256, 2433)])
def test_row_plans_match_dense(N, Ns):
    _compare(_curves(N, Ns, "fp32"), "fp32", steps=2)


# the implicit increment's tensor-core products on column-major operands, K ranges that end
# inside a chunk (M odd and even), every N they are built for
@pytest.mark.parametrize("N,Ns", [(32, 68), (64, 301), (128, 131), (256, 194)])
def test_implicit_on_columns_matches_dense(N, Ns):
    _compare(_curves(N, Ns, "fp32", scheme="implicit"), "fp32", steps=3)


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("symmetry", [0, 1, 3, 5, 7])
@pytest.mark.parametrize("adjoint", ["paper", "discrete"])
def test_column_form_options_match_dense(precision, symmetry, adjoint):
    """Both adjoints and every subspace with lambda free, an odd number of sections."""
    _compare(_curves(32, 301, precision, symmetry=symmetry, adjoint=adjoint, lambda_free=True, dtau_lambda=1e-6),
             precision)


@pytest.mark.parametrize("precision,N,Ns", [("fp64", 32, 300), ("fp32", 64, 700), ("fp32", 16, 5000)])
def test_column_form_stops_and_reports(precision, N, Ns):
    """The steps taken to a tolerance that the descent reaches part-way, the state left
    there, and the scalars of an asynchronous call that ends with an update."""
    probe = _curves(N, Ns, precision, conv="j")[1]
    J0 = probe.descend(0)["J"]
    tol = 0.5 * (J0 + probe.descend(40)["J"])
    a, b, _ = _curves(N, Ns, precision, conv="j")
    oa, ob = a.descend(40, tol), b.descend(40, tol)
    assert 0 < oa["steps"] == ob["steps"] < 40 and oa["status"] == ob["status"] == 0
    t = 1e-10 if precision == "fp64" else 5e-6
    assert rel_2(a.get_state().double().cpu().numpy(), b.get_state().double().cpu().numpy()) < t
    a.descend_async(3)
    b.descend_async(3)
    sa, sb = a.scalars(), b.scalars()
    assert sa["step"] == sb["step"] and sa["tau"] == sb["tau"] and sa["lam"] == sb["lam"]
    # |G|: the raw norm carries a_j^2, FP32 rounding of the top modes
    assert abs(sa["G_norm"] - sb["G_norm"]) <= (1e-9 if precision == "fp64" else 2e-2) * sb["G_norm"]
