"""Kernel variants chosen by size: each against the general form it stands in for.

Where a variant does the same arithmetic in another partition the results are
compared bit for bit; otherwise the tolerance is derived beside the test.
"""
import numpy as np
import pytest

import synthetic as S

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


@pytest.mark.parametrize("p", [2, 3, 4, 5, 6])
@pytest.mark.parametrize("nx,ny", [(2, 2), (3, 5), (7, 2), (12, 13)])
@pytest.mark.parametrize("riemann", [0, 1])
def test_small_tiles_equal_the_large_ones(fr, p, nx, ny, riemann):
    """Meshes of few tiles take a smaller tile shape by default; shape 1, asked for, is the large one.
    Every face and point has the same arithmetic in both: R(U) and A z agree bit for bit."""
    xe, ye = S.stretched_mesh(nx, ny, seed=p)
    X, Y = S.point_coords(xe, ye, p)
    U = _t(S.smooth_random_state(X, Y, seed=nx, amp=0.1))
    ctx = fr.Context(xe, ye, p, fr.default_opts(riemann=riemann, precond=0, m_max=1, gmres_m=1))
    z = _t(S.random_vector(U.shape, ny))
    out = []
    for tv in (0, 1):
        fr.set_launch_config(ctx, 456, tv)
        R, y = ctx.empty(), ctx.empty()
        fr.fr_residual(ctx, U, R)
        fr.fr_jv(ctx, U, R, z, 3.0, y)
        out.append((R.cpu().numpy(), y.cpu().numpy()))
    assert np.array_equal(out[0][0], out[1][0]) and np.array_equal(out[0][1], out[1][1])


@pytest.mark.parametrize("bad", [0.0, 1e-310, np.inf, np.nan])
def test_density_outside_the_normal_range_stays_visible(fr, bad):
    """A density of zero, subnormal, infinite or NaN at one point leaves the element's residual non-finite
    and the far elements' untouched."""
    p, n = 3, 9
    xe, ye = S.uniform_mesh(n)
    X, Y = S.point_coords(xe, ye, p)
    U0 = S.Vortex().state(X, Y)
    ctx = fr.Context(xe, ye, p, fr.default_opts(precond=0, m_max=1, gmres_m=1))
    R0, R = ctx.empty(), ctx.empty()
    fr.fr_residual(ctx, _t(U0), R0)
    U = U0.copy()
    U[0, 0, 5] = bad
    fr.fr_residual(ctx, _t(U), R)
    R0, R = R0.cpu().numpy(), R.cpu().numpy()
    assert not np.isfinite(R[0]).all()
    far = 4 + 4 * n
    assert np.array_equal(R[far], R0[far])
