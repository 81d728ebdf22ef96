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


@pytest.mark.parametrize("n_in,n_h,n_out", [(20, 64, 7), (21, 33, 5), (108, 256, 36), (3, 1, 2)])
@pytest.mark.parametrize("M", [1, 63, 65, 130, 1472])
def test_training_step_at_tile_edges(fr, n_in, n_h, n_out, M):
    """FP32 forward, gradients and one Adam step where 64-wide tiles, 16-deep slices, row splits and the
    16-byte loads end: against the oracle network in FP64.  A sum of K products of unit scale carries
    at most K u (u = 2^-24) relative to the sum of their magnitudes, K <= 1472: 1472 u = 9e-5, and the
    errors of a random sum grow like sqrt(K): bound 1e-5 relative in the 2-norm (the repository's)."""
    import torch
    rng = np.random.default_rng(M + n_in)
    sizes = (n_in, n_h, n_h, n_out)
    params = [(rng.standard_normal((b, a)) * np.sqrt(2.0 / a), 0.1 * rng.standard_normal(b))
              for a, b in zip(sizes[:-1], sizes[1:])]
    params = [(W.astype(np.float32).astype(np.float64), b.astype(np.float32).astype(np.float64)) for W, b in params]
    X = rng.standard_normal((M, n_in)).astype(np.float32)
    T = rng.standard_normal((M, n_out)).astype(np.float32)
    # room for other batches: the partial buffer is sized by the model, not by this call
    net = fr.MLP(n_in, n_h, n_out, max(M, 1500))
    net.set_params(fr.flat_params(params))
    Y = torch.empty((M, n_out), dtype=torch.float32, device="cuda")
    Xd, Td = _t(X), _t(T)
    net.forward(Xd, Y)
    loss = net.backward(Xd, Td)
    g = net.get_grads().astype(np.float64)
    A, Z = [X.astype(np.float64)], []
    for W, b in params:
        Z.append(A[-1] @ W.T + b)
        A.append(np.maximum(Z[-1], 0.0))
    d = (Z[2] - T) / Z[2].size
    want = [None] * 3
    for k in (2, 1, 0):
        want[k] = np.concatenate([(d.T @ A[k]).reshape(-1), d.sum(0)])
        d = (d @ params[k][0]) * (Z[k - 1] > 0) if k else d
    want = np.concatenate(want)
    assert np.linalg.norm(Y.cpu().numpy() - Z[2]) <= 1e-5 * np.linalg.norm(Z[2])
    assert abs(loss - 0.5 * np.mean((Z[2] - T) ** 2)) <= 1e-5 * abs(loss)
    assert np.linalg.norm(g - want) <= 1e-5 * np.linalg.norm(want)
    # Adam refreshes the BF16 weights: inference follows the FP32 forward to BF16 rounding
    net.adam(1e-3)
    Yb = torch.empty_like(Y)
    net.forward(Xd, Y)
    net.forward(Xd, Yb, bf16=True)
    Y, Yb = Y.cpu().numpy(), Yb.cpu().numpy()
    assert np.linalg.norm(Yb - Y) <= 3e-2 * np.linalg.norm(Y) + 1e-6


@pytest.mark.parametrize("p,prec,riemann", [(2, 0, 0), (3, 0, 1), (4, 0, 0), (2, 2, 1), (3, 1, 0), (3, 2, 0), (4, 1, 1)])
@pytest.mark.parametrize("nx,ny", [(2, 2), (5, 7), (40, 11), (61, 50)])
def test_one_launch_solve_equals_the_launches(fr, p, prec, riemann, nx, ny):
    """Small 2D Euler solves run as one launch; with a family being timed they run as the separate
    launches.  Both sum in the same order: the same iterations and the same bits, from a zero guess,
    from a nonzero one, over restarts, with both Gram-Schmidt passes forced, and for a zero
    right-hand side."""
    import torch
    xe, ye = S.stretched_mesh(nx, ny, seed=p)
    X, Y = S.point_coords(xe, ye, p)
    U = _t(S.smooth_random_state(X, Y, seed=nx, amp=0.05))
    for eta in (1.0 / 64.0, 1.0):
        ctx = fr.Context(xe, ye, p, fr.default_opts(riemann=riemann, block_precision=prec, reorth_eta=eta))
        R0 = ctx.empty()
        fr.fr_residual(ctx, U, R0)
        fr.ejacobi_factor(ctx, U, R0, 4.0)
        b, x1 = _t(S.random_vector(U.shape, 1)), _t(S.random_vector(U.shape, 2))
        for rhs, x0, m, rtol, restarts in ((b, torch.zeros_like(b), 30, 1e-8, 20), (b, 0.01 * x1, 30, 1e-7, 20),
                                           (b, torch.zeros_like(b), 3, 1e-9, 4), (b, torch.zeros_like(b), 1, 1e-3, 0),
                                           (torch.zeros_like(b), x1, 5, 1e-8, 2), (b, torch.zeros_like(b), 4, 2.0, 2)):
            res = []
            for timed in (False, True):
                x = x0.clone()
                if timed:
                    fr.fr_profile_begin(ctx, ["dots"])
                info = fr.gmres_solve(ctx, U, R0, 4.0, rhs, x, m=m, rtol=rtol, max_restarts=restarts)
                if timed:
                    fr.fr_profile_end(ctx)
                res.append((x.cpu().numpy(), info))
            assert res[0][1] == res[1][1]
            assert np.array_equal(res[0][0], res[1][0])
        ctx.close()


def test_one_launch_solve_reports_non_finite_values(fr):
    import torch
    xe, ye = S.uniform_mesh(8)
    X, Y = S.point_coords(xe, ye, 3)
    U = _t(S.Vortex().state(X, Y))
    ctx = fr.Context(xe, ye, 3)
    R0 = ctx.empty()
    fr.fr_residual(ctx, U, R0)
    fr.ejacobi_factor(ctx, U, R0, 4.0)
    b = _t(S.random_vector(U.shape, 1))
    for bad in (np.nan, np.inf):
        c = b.clone()
        c.view(-1)[17] = bad
        with pytest.raises(fr.FrError) as e:
            fr.gmres_solve(ctx, U, R0, 4.0, c, torch.zeros_like(b))
        assert e.value.code == fr.FR_ERR_NONFINITE
    x = torch.zeros_like(b)   # the context still solves
    assert fr.gmres_solve(ctx, U, R0, 4.0, b, x, rtol=1e-8).converged


def test_solves_on_several_streams_and_threads(fr):
    """Contexts on streams and threads of their own, their grids competing for the device."""
    import threading
    import torch
    cs = []
    for k in range(6):
        n, p = 20 + 7 * k, 2 + k % 3
        xe, ye = S.uniform_mesh(n)
        X, Y = S.point_coords(xe, ye, p)
        U = _t(S.Vortex(x0=0.2 * k).state(X, Y))
        cs.append((fr.Context(xe, ye, p), U, U.clone(), torch.cuda.Stream()))
    torch.cuda.synchronize()
    for ctx, U, V, s in cs:
        fr.step_row(ctx, 3, 0.05, V)
    torch.cuda.synchronize()

    def work(ctx, U, s):
        fr.step_row(ctx, 3, 0.05, U, stream=s.cuda_stream)

    ts = [threading.Thread(target=work, args=(c, U, s)) for c, U, _, s in cs]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    torch.cuda.synchronize()
    for ctx, U, V, s in cs:
        assert torch.equal(U, V)


@pytest.mark.parametrize("p,nx,ny", [(2, 3, 2), (3, 2, 5), (4, 3, 3), (5, 2, 2)])
@pytest.mark.parametrize("scale", [1.0, 30.0])
def test_fp64_block_inverse_against_the_oracle_solve(fr, p, nx, ny, scale):
    """The FP64 element blocks' inverse (panels in FP64, updates in 57-bit integers) in states whose
    variables, and so the blocks' rows and columns, differ by orders of magnitude: M^-1 r against the
    oracle's solve with its own finite-difference blocks, at the tolerance of FP64 blocks (1e-6: the
    difference quotients of step 1e-7; each side's columns carry 1e-16 / 1e-7 of the flux scale)."""
    from oracle.fr2d import Mesh
    from oracle.jfnk import ElementJacobi, Problem, element_blocks
    xe, ye = S.stretched_mesh(nx, ny, seed=p)
    X, Y = S.point_coords(xe, ye, p)
    U = S.smooth_random_state(X, Y, seed=nx, amp=0.05, base=(1.0, 0.7, -0.4, 2.0 * scale))
    ctx = fr.Context(xe, ye, p)
    fr.ejacobi_factor(ctx, _t(U), None, 30.0)
    r = S.random_vector(U.shape, 3)
    r[:, 3] *= scale
    z = ctx.empty()
    fr.ejacobi_apply(ctx, _t(r), z)
    want = ElementJacobi(element_blocks(Problem(Mesh(xe, ye), p), U, 30.0))(r)
    got = z.cpu().numpy()
    for v in range(4):
        assert np.linalg.norm(got[:, v] - want[:, v]) < 1e-6 * np.linalg.norm(want[:, v])


@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_fp64_block_inverse_keeps_non_finite_values_visible(fr, bad):
    """A non-finite state in one element makes that element's preconditioned vector non-finite."""
    xe, ye = S.uniform_mesh(6)
    X, Y = S.point_coords(xe, ye, 3)
    U = S.Vortex().state(X, Y)
    U[7, 3, 2] = bad
    ctx = fr.Context(xe, ye, 3)
    fr.ejacobi_factor(ctx, _t(U), None, 30.0)
    z = ctx.empty()
    fr.ejacobi_apply(ctx, _t(S.random_vector(U.shape, 3)), z)
    z = z.cpu().numpy()
    assert not np.isfinite(z[7]).all()
    assert np.isfinite(z[21]).all()


@pytest.mark.parametrize("n_in,n_h,n_out", [(300, 256, 100), (320, 256, 128), (108, 64, 36), (20, 33, 7), (12, 130, 120), (4, 1, 1)])
def test_network_inference_in_one_kernel_equals_the_layer_kernels(fr, n_in, n_h, n_out):
    """BF16 inference in one kernel against the layer kernels, which rows of X at an odd address and an
    output over its own input take: the same K steps, bias, rounding, so the same bits, also with
    infinities and NaN, for row counts around the 128-row tile and the number of SMs."""
    import torch
    rng = np.random.default_rng(n_in)
    most = 128 * 310 + 5
    net = fr.MLP(n_in, n_h, n_out, most)
    net.set_params(rng.standard_normal(net.nparam).astype(np.float32) * 0.1)
    X = rng.standard_normal((most, n_in)).astype(np.float32)
    X[3, 1], X[200, 0], X[201, 2] = np.inf, np.nan, -np.inf
    base = _t(np.concatenate([np.zeros(1, np.float32), X.reshape(-1)]))
    odd = base[1:].reshape(most, n_in)  # 4 bytes past a 16-byte boundary
    even = odd.clone()
    for M in (1, 127, 128, 129, 128 * 152, 128 * 153 + 1, most):
        Y = torch.full((M + 1, n_out), 7.0, dtype=torch.float32, device="cuda")
        want = torch.full((M + 1, n_out), 7.0, dtype=torch.float32, device="cuda")
        net.forward(even[:M], Y[:M], bf16=True)
        net.forward(odd[:M], want[:M], bf16=True)
        assert torch.equal(Y.view(torch.int32), want.view(torch.int32)), M
    if n_out <= n_in:  # in place: every row of X is read before Y is written
        inplace = even.clone()
        net.forward(inplace, inplace.view(-1)[:most * n_out].view(most, n_out), bf16=True)
        assert torch.equal(inplace.view(-1)[:most * n_out].view(torch.int32), want[:most].view(-1).view(torch.int32))


@pytest.mark.parametrize("p,nx,ny", [(2, 3, 2), (3, 2, 5), (4, 3, 3)])
@pytest.mark.parametrize("prec", [1, 2])
def test_reduced_precision_block_inverse_against_the_fp64_blocks(fr, p, nx, ny, prec):
    """36, 64 and 100-row blocks inverted in FP32 (panels of 16 columns in one warp's registers, the last
    panel of 4 included): M^-1 r against FP64 blocks.  FP32 elimination of n rows loses at most about
    n cond 2^-24, with cond below 1e2 at this shift: 100 * 1e2 * 6e-8 = 6e-4 < 1e-3; BF16 storage adds
    2^-9 of each entry, times cond in the worst direction of r, a few 2^-9 for a random one: 2e-2."""
    xe, ye = S.stretched_mesh(nx, ny, seed=p)
    X, Y = S.point_coords(xe, ye, p)
    U = S.smooth_random_state(X, Y, seed=nx, amp=0.05, base=(1.0, 0.7, -0.4, 2.0))
    r = S.random_vector(U.shape, 3)
    z = []
    for q in (0, prec):
        ctx = fr.Context(xe, ye, p, fr.default_opts(block_precision=q))
        fr.ejacobi_factor(ctx, _t(U), None, 30.0)
        out = ctx.empty()
        fr.ejacobi_apply(ctx, _t(r), out)
        z.append(out.cpu().numpy())
    assert np.linalg.norm(z[1] - z[0]) < (1e-3 if prec == 1 else 2e-2) * np.linalg.norm(z[0])
    U[1, 2, 3] = np.nan  # a NaN stays in its element's block
    fr.ejacobi_factor(ctx, _t(U), None, 30.0)
    fr.ejacobi_apply(ctx, _t(r), out)
    z = out.cpu().numpy()
    assert not np.isfinite(z[1]).all() and np.isfinite(z[nx * (ny // 2)]).all()
