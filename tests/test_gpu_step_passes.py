"""GPU parity of the step's row and column passes at the edges of their
ranges: every number of elements per thread on short, long and square
transforms (one pass, a smaller last radix, one thread per sequence, a
sequence within a warp and over several), several sequences per block, and
the penalisation with its coefficients everywhere, nowhere, and across the
periodic boundary of the box.  Bars per step as in test_gpu_stepper.py: the
FP64 and double-float steppers 1e-12, FP32 1e-6, relative to the oracle."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import ns2d  # noqa: E402
from paper_1804_03859_gb300 import inputs, nsstab  # noqa: E402

pytestmark = pytest.mark.gpu

TOL = {64: 1e-12, 48: 1e-12, 32: 1e-6}


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a, dtype=np.float64)).cuda()


def _rel(t, b):
    torch.cuda.synchronize()
    a = t.cpu().numpy()
    return np.linalg.norm(a - b) / np.linalg.norm(b)


def _check(st, kw, nx, ny, prec, what):
    cfg = ns2d.Config(**kw)
    w0 = inputs.wake_like_field(ny, nx, seed=41) + 0.3 * inputs.smooth_field(ny, nx, seed=42, kmax=3)
    t = _dev(w0)
    st.step_nonlinear(t, 3)
    assert _rel(t, ns2d.step_nonlinear(w0, 3, cfg)) <= 3 * TOL[prec], what
    v = inputs.gaussian_field(ny, nx, seed=43)
    out = torch.empty(ny, nx, dtype=torch.float64, device="cuda")
    st.apply_expTL(_dev(w0), _dev(v), out, 3 * cfg.dt)
    assert _rel(out, ns2d.apply_expTL(ns2d.Base.from_omega(w0, cfg), v, 3 * cfg.dt, cfg)) <= 3 * TOL[prec], what
    psi = torch.empty_like(out)
    st.stepper_poisson(_dev(v), psi)
    assert _rel(psi, ns2d.streamfunction(v, cfg)) <= TOL[prec], what


@pytest.mark.parametrize("prec", [64, 48, 32])
@pytest.mark.parametrize("nx,ny", [(8, 8), (16, 64), (64, 16), (128, 32), (256, 8), (32, 512), (1024, 16)])
def test_every_plan_at_the_edges_of_the_transform_lengths(nx, ny, prec):
    kw = dict(nx=nx, ny=ny, dt=0.01 * 128 / max(nx, 128))
    st = nsstab.Stepper(precision=prec, **kw)
    defaults = st.plans()
    _check(st, kw, nx, ny, prec, "default")
    for le in (1, 2, 3):
        for per in (1, 4):
            took = 0
            for kid in range(6):
                try:
                    st.stepper_set_plan(kid, le, per)
                    took += 1
                except nsstab.NsstabError:
                    pass
            if took:
                _check(st, kw, nx, ny, prec, (le, per))
            for kid, name in enumerate(nsstab.Stepper.KERNELS):
                st.stepper_set_plan(kid, *defaults[name])


@pytest.mark.parametrize("prec", [64, 32])
@pytest.mark.parametrize("extra", [dict(cyl_D=0.0, sponge_sigma=0.0), dict(cyl_D=0.0), dict(sponge_sigma=0.0),
                                   dict(sponge_frac=1.0), dict(cyl_x=0.0, cyl_y=0.0, cyl_D=1.2),
                                   dict(cyl_x=15.9, cyl_y=7.9, sponge_frac=0.03)])
def test_penalisation_everywhere_nowhere_and_across_the_boundary(extra, prec):
    nx, ny = 128, 64
    kw = dict(nx=nx, ny=ny, dt=0.01, **extra)
    _check(nsstab.Stepper(precision=prec, **kw), kw, nx, ny, prec, extra)


@pytest.mark.parametrize("prec", [64, 48, 32])
@pytest.mark.parametrize("nx,ny,per", [(8, 8, 1), (32, 64, 2), (256, 16, 1), (64, 32, 4)])
def test_tangent_of_both_members_in_one_launch(nx, ny, per, prec):
    """The co-integrated tangent (trajectory and perturbation in one launch
    per kernel) against the oracle's, at several pairs per block and every
    number of elements a thread."""
    kw = dict(nx=nx, ny=ny, dt=0.01 * 128 / max(nx, 128))
    cfg = ns2d.Config(**kw)
    q = inputs.wake_like_field(ny, nx, seed=51) + 0.3 * inputs.smooth_field(ny, nx, seed=52, kmax=3)
    v = inputs.gaussian_field(ny, nx, seed=53)
    T = 5 * cfg.dt
    ref = ns2d.apply_tangent(q, v, T, cfg)
    st = nsstab.Stepper(per_set=2, precision=prec, **kw)
    out = torch.empty(ny, nx, dtype=torch.float64, device="cuda")
    for le in (0, 1, 2, 3):
        if le:
            for kid in (2, 5):
                try:
                    st.stepper_set_plan(kid, le, per)
                except nsstab.NsstabError:
                    pass
        st.apply_tangent(_dev(q), _dev(v), out, T)
        assert _rel(out, ref) <= 5 * TOL[prec], (le, per)


@pytest.mark.parametrize("prec", [64, 48, 32])
@pytest.mark.parametrize("nx,ny", [(8, 8), (16, 16), (64, 32), (128, 64), (256, 128)])
def test_combined_row_passes_equal_the_separate_ones(nx, ny, prec):
    """Small grids run the inverse and the forward row pass as one kernel; a
    batch large enough to keep them apart has to give the same step, with
    selective frequency damping and without."""
    kw = dict(nx=nx, ny=ny, dt=0.01 * 128 / max(nx, 128))
    many = 608 * 16 // ny          # far beyond one block of row pairs per SM
    w0 = inputs.wake_like_field(ny, nx, seed=61) + 0.3 * inputs.smooth_field(ny, nx, seed=62, kmax=3)
    one = nsstab.Stepper(precision=prec, **kw)
    batch = nsstab.Stepper(precision=prec, per_set=many, **kw)
    a, b = _dev(w0)[None], _dev(w0)[None].repeat(many, 1, 1)
    one.step_nonlinear(a, 6)
    batch.step_nonlinear(b, 6)
    assert _rel(b[many // 2], a[0].cpu().numpy()) <= 6 * TOL[prec]
    a, b = _dev(w0)[None], _dev(w0)[None].repeat(many, 1, 1)
    one.sfd_baseflow(a, chi=0.5, Delta=1.0, tol=0.0, max_steps=6, check_every=3)
    batch.sfd_baseflow(b, chi=0.5, Delta=1.0, tol=0.0, max_steps=6, check_every=3)
    assert _rel(b[-1], a[0].cpu().numpy()) <= 6 * TOL[prec]
