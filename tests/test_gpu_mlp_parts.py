"""Weight gradients of batches of more than one part of rows (4096 rows each), whose partial sums go
through a buffer and a kernel of their own."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,most", [(4096, 4096), (4097, 4097), (8192, 8192), (8193, 12300), (12300, 12300), (100, 9000)])
@pytest.mark.parametrize("n_in,n_h,n_out", [(20, 64, 8), (21, 33, 5)])
def test_gradients_over_several_parts(n_in, n_h, n_out, M, most):
    """Around the ends of a part, with room for more rows than the call has, and a second call after one
    of other rows: gradients against FP64.  A sum of K terms in FP32 with random signs carries about
    u sqrt(K / 2) of itself (u = 2^-24, K = 4096 in a chain): 3e-6, bound 1e-5 in the 2-norm."""
    import torch
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    import paper_1904_04825_gb300 as fr
    rng = np.random.default_rng(M + n_in)
    sizes = (n_in, n_h, n_h, n_out)
    params = [((rng.standard_normal((b, a)) * np.sqrt(2.0 / a)).astype(np.float32).astype(np.float64),
               (0.1 * rng.standard_normal(b)).astype(np.float32).astype(np.float64)) for a, b in zip(sizes[:-1], sizes[1:])]
    net = fr.MLP(n_in, n_h, n_out, most)
    net.set_params(fr.flat_params(params))
    for rows in (most, M):
        X = rng.standard_normal((rows, n_in)).astype(np.float32)
        T = rng.standard_normal((rows, n_out)).astype(np.float32)
        Xd, Td = torch.from_numpy(X).cuda(), torch.from_numpy(T).cuda()
        net.forward(Xd, torch.empty((rows, n_out), dtype=torch.float32, device="cuda"))
        net.backward(Xd, Td)
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
        for k, w in enumerate(want):
            o = sum(v.size for v in want[:k])
            assert np.linalg.norm(g[o:o + w.size] - w) <= 1e-5 * np.linalg.norm(w), (rows, k)
