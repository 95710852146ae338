"""The dense SR solve where diagonal entries of S are exact powers of four: without a
shift, S_ii = 1 - m^2 of a spin whose samples sum to zero is 1, and of a shift of 3
it is 4.  First and interior pivots, one and more panels, both precisions.

Tolerance as in test_dense_solve_gpu: a backward-stable solve of order n leaves
||A x - b|| <= c n u (||A|| ||x|| + ||b||), u = 2^-53; 8 n u."""
import numpy as np
import pytest
import torch

from paper_2112_10526_gb300 import inputs as I
from paper_2112_10526_gb300 import nk
from gpu_util import cu, dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["f64", "mixed"])
@pytest.mark.parametrize("eps", [0.0, 3.0])
@pytest.mark.parametrize("spins", [[0], [2], [0, 1, 3]])
@pytest.mark.parametrize("N,M,Ns", [(7, 6, 256), (9, 11, 1024)])
def test_spins_of_zero_mean(N, M, Ns, spins, eps, prec):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    p = I.rbm_params(N, M, 3, 0.3)
    s = I.random_configs(Ns, N, 5)
    g = np.random.default_rng(11)
    for i in spins:
        s[:, i] = g.permutation(np.repeat(np.array([1, -1], dtype=np.int8), Ns // 2))
    sd = s.astype(np.float64)
    T = np.tanh(p[N:N + M] + sd @ p[N + M:].reshape(M, N).T)
    J = np.concatenate([sd, T, (T[:, :, None] * sd[:, None, :]).reshape(Ns, -1)], 1)
    J -= J.mean(0)
    F = J.T @ np.random.default_rng(7).normal(size=Ns) * (2.0 / Ns)
    A = J.T @ J / Ns + eps * np.eye(p.size)
    assert all(A[i, i] == 1.0 + eps for i in spins)
    with nk.Ctx() as ctx:
        delta = torch.empty(p.size, dtype=torch.float64, device=dev())
        nk.nk_sr_solve(ctx, cu(p), N, M, cu(s), cu(F), delta, solver="cholesky", diag_shift=eps, precision=prec)
        x = delta.cpu().numpy()
    n = max(p.size, Ns)
    size = np.linalg.norm(A) * np.linalg.norm(x)
    assert np.linalg.norm(A @ x - F) <= 8 * n * 2.0 ** -53 * (size + np.linalg.norm(F))
