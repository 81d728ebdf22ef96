"""Solves of small 2D Euler contexts that run as one launch: where they hand over to the
separate launches, and how they end when a bounded wait gave up."""
import numpy as np
import pytest

import synthetic as S
from oracle.fr2d import Mesh
from oracle.jfnk import Problem
from oracle.steppers import PtcOpts, SolverOpts
from oracle.steppers import step_bdf2 as o_bdf2
from oracle.steppers import step_esdirk as o_esdirk
from oracle.steppers import step_row as o_row
from oracle.tableaus import ESDIRK, ROW

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def fr():
    import torch
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    import paper_1904_04825_gb300 as mod
    return mod


def _t(a):
    import torch
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def _rel(a, b):
    return np.linalg.norm(a - b) / np.linalg.norm(b)


@pytest.mark.parametrize("m", [58, 59, 60, 63])
@pytest.mark.parametrize("stepper", ["row", "esdirk", "bdf2"])
def test_steps_around_the_longest_restart_of_one_launch(fr, m, stepper):
    """One launch holds the partial sums of up to 58 basis vectors; longer restarts, the paper's 60
    among them, take the separate launches, which add to the guess they are given.  The second and
    later solves find the last solution in that buffer: steps against the oracle, at the tolerance
    of the repository's stepper tests (1e-9 with solves to 1e-12)."""
    p = 2
    xe, ye = S.uniform_mesh(6)
    X, Y = S.point_coords(xe, ye, p)
    U0 = S.Vortex().state(X, Y)
    prob = Problem(Mesh(xe, ye), p)
    tight = SolverOpts(tol_lin=1e-12, m=m, max_restarts=40)
    ctx = fr.Context(xe, ye, p, fr.default_opts(tol_lin=1e-12, m_max=m, gmres_m=m, gmres_max_restarts=40))
    po, oo = fr.default_ptc_opts(tol_nl=1e-12, tol_lin=1e-3), PtcOpts(tol_nl=1e-12, tol_lin=1e-3)
    U, Uo = _t(U0), U0.copy()
    if stepper == "row":
        for _ in range(2):
            assert fr.step_row(ctx, 3, 0.1, U).converged
            Uo, _s = o_row(prob, ROW[3](), 0.1, Uo, tight)
    elif stepper == "esdirk":
        assert fr.step_esdirk(ctx, 3, 0.1, U, po).converged
        Uo, _s = o_esdirk(prob, ESDIRK[3](), 0.1, Uo, oo, tight)
    else:
        Up, Upo = ctx.empty(), None
        for k in range(2):
            assert fr.step_bdf2(ctx, 0.1, U, Up, k == 0, po).converged
            Uo, Upo, _s = o_bdf2(prob, 0.1, Uo, Upo, k == 0, oo, tight)
    assert _rel(U.cpu().numpy(), Uo) < 1e-9
    ctx.close()


@pytest.mark.parametrize("prec", [0, 1, 2])
def test_flag_of_an_earlier_wait_reaches_the_next_solve(fr, prec):
    """A wait of the apply that gave up sets the context's flag: the next solve, and every later one
    and every step, reports it, although their own waits end."""
    import torch
    p = 2
    xe, ye = S.uniform_mesh(8)
    X, Y = S.point_coords(xe, ye, p)
    U = _t(S.Vortex().state(X, Y))
    ctx = fr.Context(xe, ye, p, fr.default_opts(block_precision=prec))
    R0, z = ctx.empty(), ctx.empty()
    fr.fr_residual(ctx, U, R0)
    fr.ejacobi_factor(ctx, U, R0, 20.0)
    b = _t(S.random_vector(ctx.shape, 3))
    assert fr.gmres_solve(ctx, U, R0, 20.0, b, torch.zeros_like(b)).converged
    fr.fr_set_wait_test(ctx, polls=2000, skip_first_copy=True)
    fr.ejacobi_apply(ctx, b, z)
    fr.fr_set_wait_test(ctx)
    for _ in range(2):
        with pytest.raises(fr.FrError) as e:
            fr.gmres_solve(ctx, U, R0, 20.0, b, torch.zeros_like(b))
        assert e.value.code == fr.FR_ERR_TIMEOUT
    with pytest.raises(fr.FrError) as e:
        fr.step_row(ctx, 2, 0.05, U)
    assert e.value.code == fr.FR_ERR_TIMEOUT
    torch.cuda.synchronize()
    ctx.close()


@pytest.mark.parametrize("prec,nx,ny", [(0, 61, 50), (2, 40, 11)])
def test_grid_barrier_runs_out_and_the_context_keeps_saying_so(fr, prec, nx, ny):
    """With a limit of a few looks the CTAs without a tile give up at the grid barrier: the solve
    returns FR_ERR_TIMEOUT, and so does every later one of that context, with the default limit too.
    Another context then solves as before."""
    import torch
    p = 3
    xe, ye = S.uniform_mesh(nx)[0], S.uniform_mesh(ny)[1]
    X, Y = S.point_coords(xe, ye, p)
    U = _t(S.smooth_random_state(X, Y, seed=nx, amp=0.05))
    b = _t(S.random_vector(U.shape, 3))

    def context():
        ctx = fr.Context(xe, ye, p, fr.default_opts(block_precision=prec))
        R0 = ctx.empty()
        fr.fr_residual(ctx, U, R0)
        fr.ejacobi_factor(ctx, U, R0, 20.0)
        return ctx, R0

    ctx, R0 = context()
    want = torch.zeros_like(b)
    assert fr.gmres_solve(ctx, U, R0, 20.0, b, want).converged
    for polls in (1, 0, 0):
        fr.fr_set_wait_test(ctx, polls=polls)
        with pytest.raises(fr.FrError) as e:
            fr.gmres_solve(ctx, U, R0, 20.0, b, torch.zeros_like(b))
        assert e.value.code == fr.FR_ERR_TIMEOUT
    torch.cuda.synchronize()
    ctx.close()
    ctx, R0 = context()
    x = torch.zeros_like(b)
    assert fr.gmres_solve(ctx, U, R0, 20.0, b, x).converged
    assert torch.equal(x, want)
    ctx.close()


_FIRST_SOLVES = """
import hashlib, sys, threading
sys.path.insert(0, sys.argv[1])
import torch
import paper_1904_04825_gb300 as fr
import synthetic as S
cs = []
for k in range(6):
    xe, ye = S.uniform_mesh(10 + k)
    U = torch.from_numpy(S.Vortex().state(*S.point_coords(xe, ye, 3))).cuda()
    cs.append((fr.Context(xe, ye, 3, fr.default_opts(block_precision=k % 3, riemann=k // 3)), U, torch.cuda.Stream()))
torch.cuda.synchronize()
gate = threading.Barrier(6)
def work(ctx, U, s):
    gate.wait()
    fr.step_row(ctx, 3, 0.05, U, stream=s.cuda_stream)
if sys.argv[2] == "threads":
    ts = [threading.Thread(target=work, args=c) for c in cs]
    [t.start() for t in ts]
    [t.join() for t in ts]
else:
    for ctx, U, s in cs:
        fr.step_row(ctx, 3, 0.05, U, stream=s.cuda_stream)
torch.cuda.synchronize()
print([hashlib.sha1(U.cpu().numpy().tobytes()).hexdigest() for _, U, _ in cs])
"""


def test_first_solves_of_a_process_on_several_threads():
    """The grid's size is found by the first solve of a process: six threads that solve first, together,
    end with the bits of one thread after another."""
    import os
    import subprocess
    import sys
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    out = [subprocess.run([sys.executable, "-c", _FIRST_SOLVES, root, how], capture_output=True, text=True, timeout=300)
           for how in ("threads", "in turn")]
    assert out[0].returncode == 0 and out[1].returncode == 0, out[0].stderr + out[1].stderr
    assert out[0].stdout == out[1].stdout


def test_autotune_times_the_form_that_solves_take(fr):
    """Thirteen configurations of two cycles: two launches each and a few where the solves run as one
    launch; with a restart length that does not fit, and on a batch's instance, dozens per cycle."""
    p, m = 2, 30
    xe, ye = S.uniform_mesh(12)
    U = _t(S.Vortex().state(*S.point_coords(xe, ye, p)))

    def launches(ctx):
        n = fr.fr_kernel_launches()
        vb, tv, best, default = fr.autotune(ctx, U, 20.0, reps=1)
        assert 0.0 < best <= default
        return fr.fr_kernel_launches() - n

    assert 13 * 2 <= launches(fr.Context(xe, ye, p, fr.default_opts(gmres_m=m))) <= 13 * 2 + 10
    assert launches(fr.Context(xe, ye, p, fr.default_opts(m_max=60, gmres_m=60))) > 13 * 2 * 60
    B = fr.Batch([(xe, ye)], [p], fr.default_opts(gmres_m=m))
    assert launches(B.members[0]) > 13 * 2 * m


def test_solve_that_turns_non_finite_in_a_later_cycle_reports_the_earlier_ones(fr):
    """On cells 1e100 wide ||x||^2 overflows, so the second cycle's difference step is zero and its
    residual b - shift x, 1.10 ||b|| here (by the oracle); with ||b|| = 1.28e154, whose square is below
    1.8e308, that one's square is not: one launch reports what the separate launches do, the first
    cycle's iterations and residual."""
    import ctypes
    import torch
    p, m, scale = 2, 10, 1e100
    xe, ye = S.uniform_mesh(6)
    U = _t(S.Vortex().state(*S.point_coords(xe, ye, p)))
    ctx = fr.Context(xe * scale, ye * scale, p)
    R0 = ctx.empty()
    fr.fr_residual(ctx, U, R0)
    fr.ejacobi_factor(ctx, U, R0, 1.0 / scale)
    b = S.random_vector(tuple(U.shape), 1)
    b = _t(b * (1.28e154 / np.linalg.norm(b)))
    infos = []
    for timed in (False, True):
        if timed:
            fr.fr_profile_begin(ctx, ["dots"])
        x, info = torch.zeros_like(b), fr.fr_gmres_info()
        rc = fr.lib.gmres_solve(ctx.handle, U.data_ptr(), R0.data_ptr(), 1.0 / scale, b.data_ptr(), x.data_ptr(), m, 1e-12,
                                5, ctypes.byref(info), None)
        assert rc == fr.FR_ERR_NONFINITE
        infos.append((info.iters, info.restarts, info.converged, info.relres))
    fr.fr_profile_end(ctx)
    assert infos[0] == infos[1] and infos[0][0] == m
    ctx.close()
