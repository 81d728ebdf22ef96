"""Device functions of the library alone, through tests/device_checks.cu (built here with the
library's own flags), where the entry points cannot reach the cases that matter."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

import synthetic as S
from oracle.fr2d import Mesh, roe, rusanov
from oracle.jfnk import Problem, element_blocks

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dev(tmp_path_factory):
    import torch
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    from paper_1904_04825_gb300 import _build as B
    out = str(tmp_path_factory.mktemp("dev") / "device_checks.so")
    src = os.path.join(os.path.dirname(os.path.abspath(__file__)), "device_checks.cu")
    r = subprocess.run([B.nvcc(), *B.ARCH, *B.FLAGS, "-shared", src, "-o", out], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    return ctypes.CDLL(out)


def _dp(a):
    assert a.dtype == np.float64 and a.flags.c_contiguous
    return a.ctypes.data_as(ctypes.POINTER(ctypes.c_double))


def _inverse(dev, M):
    M, out = np.ascontiguousarray(M), np.empty(M.shape)
    assert dev.fp64_inverse(len(M), _dp(M), _dp(out)) == 0
    return out


def _exact_inverse(M):
    """Gauss-Jordan in extended precision, pivots by scaled rows."""
    n, A = len(M), np.concatenate([M, np.eye(len(M))], 1).astype(np.longdouble)
    for c in range(n):
        q = c + int(np.argmax(np.abs(A[c:, c]) / np.abs(A[c:, :n]).max(1)))
        A[[c, q]] = A[[q, c]]
        A[c] /= A[c, c]
        f = A[:, c].copy()
        f[c] = 0
        A -= f[:, None] * A[c]
    return A[:, n:]


@pytest.mark.parametrize("n", [36, 40, 64, 100, 135, 144])
def test_fp64_block_inverse_at_every_width(dev, n):
    """Widths whose rows, two threads each up to 100, end inside a warp and whose last panel is 4, 7, 8
    or 16 columns wide.  M = 4 I + G, G of entries N(0, 1/n): cond below 10, so n u cond = 144 * 1.1e-16
    * 10 = 1.6e-13 per entry, relative to the largest."""
    M = 4.0 * np.eye(n) + np.random.default_rng(n).standard_normal((n, n)) / np.sqrt(n)
    want = _exact_inverse(M)
    assert np.abs(_inverse(dev, M) - want).max() < 1.6e-13 * np.abs(want).max()


@pytest.mark.parametrize("case", ["unit", "thin cells", "SI, shift 1e6", "SI, shift 1e4", "units far apart"])
@pytest.mark.parametrize("p", [2, 3, 4, 5])
def test_fp64_block_inverse_of_badly_scaled_blocks(dev, p, case):
    """M^-1 r of the oracle's element blocks, variable by variable, against the exact inverse: cells 1e-4
    thin, air in SI units on centimetre cells (density 1.2, speed of sound 340, energy 2e5), and variables
    in units that differ by 2^27, 2^-17 and 2^40.  One-pivot-at-a-time elimination in FP64
    with the same pivot rule, emulated on the CPU, leaves up to 5e-13 (SI, p = 2, where pivots fall
    across variables): bound 1e-12.  Powers of two change no rounding but the choice of pivots (1e-11
    in the emulation at p = 2): bound 1e-10 there."""
    xe, ye = S.stretched_mesh(3, 2, seed=p)
    base = dict(seed=3, amp=0.05, base=(1.0, 0.7, -0.4, 2.0))
    if case == "thin cells":
        X, Y = S.point_coords(xe, np.array([0.0, 1.0, 2.0]), p)
        M = element_blocks(Problem(Mesh(xe, np.array([0.0, 1e-4, 2e-4])), p), S.smooth_random_state(X, Y, **base), 30.0)[0]
    else:
        X, Y = S.point_coords(xe, ye, p)
        U = S.smooth_random_state(X, Y, **base)
        if case.startswith("SI"):
            U = U * (1.2 * np.array([1.0, 290.0, 290.0, 290.0**2]))[None, :, None]
            M = element_blocks(Problem(Mesh(0.01 * xe, 0.01 * ye), p), U, float(case.split()[-1]))[0]
        else:
            M = element_blocks(Problem(Mesh(xe, ye), p), U, 30.0)[0]
    n, npt = len(M), (p + 1) ** 2
    rng = np.random.default_rng(p)
    if case == "units far apart":
        d = np.repeat(np.exp2([0, 27, -17, 40]), npt)
        M = d[:, None] * M / d
    want, got = _exact_inverse(M), _inverse(dev, M)
    size = [float(np.median(np.abs(want[v * npt:(v + 1) * npt, v * npt:(v + 1) * npt]))) for v in range(4)]
    for _ in range(4):
        r = rng.standard_normal(n) / np.repeat(size, npt)
        z, err = want @ r, (got - want) @ r
        for v in range(4):
            k = slice(v * npt, (v + 1) * npt)
            assert np.linalg.norm(err[k]) < (1e-10 if case == "units far apart" else 1e-12) * np.linalg.norm(z[k])


@pytest.mark.parametrize("bad", [np.nan, np.inf, -np.inf])
def test_fp64_block_inverse_of_non_finite_blocks(dev, bad):
    """A non-finite entry spreads over the inverse instead of vanishing in an integer."""
    M = 4.0 * np.eye(64) + np.random.default_rng(1).standard_normal((64, 64)) / 8.0
    M[17, 40] = bad
    assert not np.isfinite(_inverse(dev, M)).all()


@pytest.mark.parametrize("nblk", [1, 2, 19, 32])
def test_grid_barrier_over_the_wrap_of_its_counter(dev, nblk):
    """The counter of a long solve wraps: rounds that begin at zero, below 2^32 and below 2^31 (where
    the difference of signed values would turn) all separate the notes before from those behind, and
    carry the done bit."""
    for start in (0, 2**32 - 40 * nblk, 2**31 - 40 * nblk):
        assert dev.check_barrier(nblk, ctypes.c_uint(start), 60) == 0


@pytest.mark.parametrize("kind", [0, 1])
@pytest.mark.parametrize("direction", [0, 1])
@pytest.mark.parametrize("jump", [0.3, 1e-3])
def test_common_flux_is_as_accurate_as_with_the_full_operations(dev, kind, direction, jump):
    """The common flux of R(U) and A z (reciprocals and roots by one step from the approximate units,
    both sides' fluxes summed undivided) against the extended-precision flux: per variable, its rms error
    is no larger than that of the IEEE form of the element blocks.  The two share most of their roundings;
    the ratio of two rms errors over n samples scatters by less than 1 / sqrt(2 n) = 0.16 % for n = 2e5:
    bound 1 + 3 * 0.0016."""
    n = 200_000
    rng = np.random.default_rng(7)
    rho, u, v, p = rng.uniform(0.5, 2.0, n), rng.normal(0, 1.0, n), rng.normal(0, 1.0, n), rng.uniform(0.5, 6.0, n)
    qm = S.conserved(rho, u, v, p)
    d = jump * rng.uniform(-1.0, 1.0, (4, n))
    qp = S.conserved(rho * (1.0 + d[0]), u + d[1], v + d[2], p * (1.0 + d[3]))
    fast, full = np.empty_like(qm), np.empty_like(qm)
    assert dev.fluxes(n, _dp(qm), _dp(qp), kind, direction, _dp(fast), _dp(full)) == 0
    exact = (roe if kind else rusanov)(qm.T.astype(np.longdouble), qp.T.astype(np.longdouble), direction, np.longdouble(1.4))
    rms = [np.sqrt(np.mean((f.T - exact) ** 2, axis=1)) for f in (fast, full)]
    assert (rms[0] <= 1.005 * rms[1]).all(), rms[0] / rms[1]


def test_fast_reciprocal_and_root(dev):
    """One step of third order from the approximate units.  1 / x: the approximation is within 2^-19.9, the
    step leaves 2^-59.7 of x, so the rounding is right except within 1/100 of the last place of a tie:
    one unit at most, in fewer than 1e-3 of the arguments.  The root starts from a rounded x r, whose error
    enters with half its size: at most 1/2 + 1/4 units and the step's 2^-59, so one unit at most, less
    often than in a quarter.  Arguments at the ends of the range and beyond take the full operations."""
    n = 1 << 24
    out = (ctypes.c_ulonglong * 4)()
    assert dev.rcp_sqrt(n, out) == 0
    assert out[0] <= 1 and out[1] <= 1e-3 * n
    assert out[2] <= 1 and out[3] <= 0.25 * n
    tiny, big = np.finfo(np.float64).tiny, np.finfo(np.float64).max
    x = np.array([0.0, -0.0, np.inf, -np.inf, np.nan, 5e-324, tiny / 2, tiny, big, -big, -1.0, -tiny, 2.0**-974, 2.0**962,
                  2.0**-975, 2.0**961])
    got = np.empty((2, x.size))
    assert dev.rcp_sqrt_at(x.size, _dp(x), _dp(got)) == 0
    with np.errstate(divide="ignore", invalid="ignore", over="ignore"):
        assert np.array_equal(got[0], 1.0 / x, equal_nan=True)
        assert np.array_equal(got[1], np.sqrt(x), equal_nan=True)


def test_larger_wave_speed_ignores_a_nan_of_either_sign(dev):
    """The larger of two non-negative values by their bit patterns gives what fmax gives, whatever the
    sign bit of a NaN (the root of a negative pressure comes with it set)."""
    neg_nan = np.copysign(np.nan, -1.0)
    v = [0.0, 5e-324, 1e-300, 1.0, np.nextafter(1.0, 2.0), 3.5, 1e300, np.inf, np.nan, neg_nan]
    a, b = (np.ascontiguousarray(m.ravel()) for m in np.meshgrid(np.array(v), np.array(v)))
    out = np.empty_like(a)
    assert dev.max_nonneg(a.size, _dp(a), _dp(b), _dp(out)) == 0
    assert np.array_equal(out, np.fmax(a, b), equal_nan=True)


@pytest.mark.parametrize("p", [2, 3])
@pytest.mark.parametrize("dim", [2, 3])
def test_negative_pressure_on_one_side_of_a_face(monkeypatch, dim, p):
    """An element whose pressure is negative has no speed of sound; the faces to its neighbours take the
    neighbours' wave speed, as fmax does: R(U) equals the oracle's with fmax, to its 1e-12."""
    import torch
    import oracle.fr3d
    import paper_1904_04825_gb300 as fr
    opts = fr.default_opts(precond=0, m_max=1, gmres_m=1)
    if dim == 2:
        xe, ye = S.stretched_mesh(5, 4, seed=p)
        U = S.smooth_random_state(*S.point_coords(xe, ye, p), seed=1, amp=0.05)
        ctx = fr.Context(xe, ye, p, opts)
    else:
        e = S.stretched_mesh3d(4, 3, 5, seed=p)
        U = S.TaylorGreen().state(*S.point_coords3d(*e, p))
        ctx = fr.Context3D(*e, p, opts)
    kin = 0.5 * (U[7, 1:-1] ** 2).sum(0) / U[7, 0]
    U[7, -1] = kin - 0.3 * (U[7, -1] - kin)  # pressure times -0.3
    R = ctx.empty()
    fr.fr_residual(ctx, torch.from_numpy(U).cuda(), R)
    R = R.cpu().numpy()
    with monkeypatch.context() as m, np.errstate(invalid="ignore"):
        m.setattr(np, "maximum", np.fmax)  # the oracle's wave speed
        want = (Problem(Mesh(xe, ye), p).R(U) if dim == 2 else
                oracle.fr3d.residual3d(U, oracle.fr3d.Mesh3D(*e), p, oracle.fr3d.Gas3D(mu=0.0)))
    assert np.isfinite(want).all()
    assert np.linalg.norm(R - want) < 1e-12 * np.linalg.norm(want)
