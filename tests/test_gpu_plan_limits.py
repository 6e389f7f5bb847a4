"""Grids at the limits of the launch plans: rows and columns of 4096 points
beside very short ones, where a default plan, a plan derived from it or the
common plan of a ragged batch is close to the largest block or the largest
shared memory a kernel can have."""
import os
import subprocess
import sys

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import krylov, ns2d  # noqa: E402
from paper_1804_03859_gb300 import inputs, nsstab  # noqa: E402

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a, dtype=np.float64)).cuda()


def _rel(t, b):
    torch.cuda.synchronize()
    a = t.cpu().numpy()
    return np.linalg.norm(a - b) / np.linalg.norm(b)


@pytest.mark.parametrize("grids", [[(4096, 8)], [(4096, 8), (128, 64)], [(1024, 16), (64, 32)], [(512, 16), (32, 32)]])
def test_persistent_serving_of_long_rows_and_of_small_grids_beside_them(grids):
    """One 4-step Arnoldi factorisation per grid in one persistent launch.
    A row of 4096 points fills a block by itself, and the small grid's rows
    do not fill a whole number of the blocks it shares the launch with.  The
    Ritz values move by less than the relative error of the products (0.02
    to 0.2 of it, from perturbed products of the oracle), so the bar is the
    FP32 step's, 1e-6 a step."""
    T, m, nev = 0.005, 4, 2
    jobs, steps = [], []
    for i, (nx, ny) in enumerate(grids):
        dt = min(T, 0.01 * 128 / nx)
        steps.append(round(T / dt))
        jobs.append(dict(nx=nx, ny=ny, dt=dt, Re=50.0, cyl_D=1.0, base=_dev(inputs.wake_like_field(ny, nx, seed=5 + i)),
                         v0=_dev(inputs.gaussian_field(ny, nx, seed=15 + i))))
    rc, res, nwaves = nsstab.serve_eigs(jobs, m=m, nev=nev, tol=1e-6, T=T, max_restarts=0, precision=32, persistent=True)
    assert rc == nsstab.NOT_CONVERGED and nwaves == 1
    for j, r, n in zip(jobs, res, steps):
        cfg = ns2d.Config(nx=j["nx"], ny=j["ny"], dt=j["dt"], Re=50.0, cyl_D=1.0)
        b = ns2d.Base.from_omega(j["base"].cpu().numpy(), cfg)
        ref = krylov.arnoldi_eigs(lambda x: ns2d.apply_expTL(b, x.reshape(cfg.ny, cfg.nx), T, cfg).ravel(),
                                  j["v0"].cpu().numpy().ravel(), m=m, nev=nev, tol=1e-6)
        assert r["n_matvec"] == m and len(r["mu"]) == len(ref.mu)
        assert np.abs(r["mu"] - ref.mu).max() <= n * 1e-6


# The double-float stepper's 1e-12 a step holds at a spacing of 1/32 (512x256):
# the differences of psi lose one more bit with every halving of the finer one.
def _step_tol(prec, cfg):
    return 1e-12 if prec == 64 else 1e-12 / 32 / min(cfg.Lx / cfg.nx, cfg.Ly / cfg.ny)


@pytest.mark.parametrize("prec", [64, 48])
@pytest.mark.parametrize("nx,ny,members", [(4096, 8, 1), (4096, 16, 2), (4096, 32, 1), (8, 4096, 4), (16, 4096, 1),
                                           (32, 4096, 1)])
def test_steppers_of_few_long_sequences(nx, ny, members, prec):
    """Few sequences ask for few elements a thread, 4096 points for many."""
    kw = dict(nx=nx, ny=ny, dt=0.01 / 32)
    cfg = ns2d.Config(**kw)
    st = nsstab.Stepper(precision=prec, per_set=members, **kw)
    w0 = inputs.wake_like_field(ny, nx, seed=71) + 0.3 * inputs.smooth_field(ny, nx, seed=72, kmax=3)
    t = _dev(np.stack([w0] * members))
    st.step_nonlinear(t, 3)
    ref = ns2d.step_nonlinear(w0, 3, cfg)
    v = inputs.gaussian_field(ny, nx, seed=73)
    out = torch.empty_like(t)
    st.apply_expTL(_dev(w0), _dev(np.stack([v] * members)), out, 3 * cfg.dt)
    lin = ns2d.apply_expTL(ns2d.Base.from_omega(w0, cfg), v, 3 * cfg.dt, cfg)
    for k in range(members):
        assert _rel(t[k], ref) <= 3 * _step_tol(prec, cfg)
        assert _rel(out[k], lin) <= 3 * _step_tol(prec, cfg)


TANGENT = """
import sys
import numpy as np, torch
from oracle import ns2d
from paper_1804_03859_gb300 import inputs, nsstab
nx, ny, le, per = map(int, sys.argv[1:])
kw = dict(nx=nx, ny=ny, dt=0.01 * 128 / nx)
cfg = ns2d.Config(**kw)
q = inputs.wake_like_field(ny, nx, seed=81) + 0.3 * inputs.smooth_field(ny, nx, seed=82, kmax=3)
v = inputs.gaussian_field(ny, nx, seed=83)
st = nsstab.Stepper(per_set=2, precision=32, **kw)
if le:
    st.stepper_set_plan(2, le, per)
out = torch.empty(ny, nx, dtype=torch.float64, device="cuda")
st.apply_tangent(torch.from_numpy(q).cuda(), torch.from_numpy(v).cuda(), out, 5 * cfg.dt)
torch.cuda.synchronize()
ref = ns2d.apply_tangent(q, v, 5 * cfg.dt, cfg)
err = np.linalg.norm(out.cpu().numpy() - ref) / np.linalg.norm(ref)
assert err <= 5 * 1e-6, err
"""


@pytest.mark.parametrize("nx,ny,le,per", [(2048, 64, 0, 0), (2048, 8, 0, 0), (4096, 32, 0, 0), (512, 64, 2, 4),
                                          (2048, 32, 1, 1)])
def test_fp32_tangent_needs_no_other_stepper_in_the_process(nx, ny, le, per):
    """The right-hand side of the FP32 tangent runs at more elements a thread
    than the plan it comes from, with up to 139 KB of shared memory: in a
    process of its own, where no other stepper raised a kernel's limit.  Bar
    as in test_gpu_step_passes.py, 1e-6 a step."""
    r = subprocess.run([sys.executable, "-c", TANGENT, *map(str, (nx, ny, le, per))], cwd=ROOT, capture_output=True,
                       text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-800:]


@pytest.mark.parametrize("nx,ny", [(512, 64), (512, 32)])
def test_autotuned_plans_are_no_slower_than_the_default_ones(nx, ny):
    """On small grids the step runs row passes in pairs, as one kernel or as
    two, so the plans have to be chosen by what the step launches.  Double-float,
    tuned eight times, 5% over the default step at most (repeated steps differ by
    1%; chosen from the separate kernels' launches, one tuning in four was 5 to
    11% slower)."""
    dt, n = 0.01 * 128 / nx, 200
    st = nsstab.Stepper(nx=nx, ny=ny, dt=dt, precision=48)
    v = _dev(inputs.gaussian_field(ny, nx, seed=92))
    out = torch.empty_like(v)
    st.apply_expTL(_dev(inputs.wake_like_field(ny, nx, seed=91)), v, out, dt)

    def step_time():
        e = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
        best = float("inf")
        for _ in range(8):
            e[0].record()
            st.apply_expTL(None, v, out, n * dt)
            e[1].record()
            e[1].synchronize()
            best = min(best, e[0].elapsed_time(e[1]))
        return best

    default = step_time()
    for _ in range(8):
        st.stepper_autotune()
        assert step_time() <= 1.05 * default, st.plans()
