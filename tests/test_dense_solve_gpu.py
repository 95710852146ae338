"""The direct SR solvers at the edges of their blocks (panels of 64, tiles of
128 x 32, chunks of 64 samples, the sizes from which S takes the tensor cores),
in both precisions, by the residual of the system.

Tolerance: a backward-stable Cholesky solve of order n leaves ||A x - b|| <=
c n u (||A|| ||x|| + ||b||) with u = 2^-53 and a small c; forming S from its
factors adds the same again.  8 n u is used, also for diag_shift = 1e-9, where S
+ eps I is nearly singular and only the FP64 path promises it."""
import numpy as np
import pytest
import torch

from paper_2112_10526_gb300 import inputs as I
from paper_2112_10526_gb300 import nk
from gpu_util import cu, dev

pytestmark = pytest.mark.gpu

# Np = 63, 64, 66, 287, 577, 577, 577, 1055
SIZES = [(3, 15, 40), (4, 12, 64), (7, 7, 65), (15, 17, 129), (16, 33, 64), (16, 33, 65), (16, 33, 1000),
         (31, 32, 200)]


@pytest.fixture(scope="module")
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    with nk.Ctx() as c:
        yield c


def _system(N, M, Ns):
    p = I.rbm_params(N, M, 3, 0.3)
    s = I.random_configs(Ns, N, 5)
    sd = s.astype(np.float64)
    T = np.tanh(p[N:N + M] + sd @ p[N + M:].reshape(M, N).T)
    J = np.concatenate([sd, T, (T[:, :, None] * sd[:, None, :]).reshape(Ns, -1)], 1)
    J -= J.mean(0)
    F = J.T @ np.random.default_rng(7).normal(size=Ns) * (2.0 / Ns)
    return p, s, J.T @ J / Ns, F


@pytest.mark.parametrize("solver", ["cholesky", "cholesky_samplespace"])
@pytest.mark.parametrize("prec,eps", [("f64", 0.01), ("mixed", 0.01), ("f64", 1e-9)])
@pytest.mark.parametrize("N,M,Ns", SIZES)
def test_direct_solve_residual(ctx, N, M, Ns, prec, eps, solver):
    if solver == "cholesky_samplespace" and eps < 1e-6:
        pytest.skip("the sample-space form divides by eps: it is not backward stable for the parameter-space system")
    p, s, S, F = _system(N, M, Ns)
    delta = torch.empty(p.size, dtype=torch.float64, device=dev())
    nk.nk_sr_solve(ctx, cu(p), N, M, cu(s), cu(F), delta, solver=solver, diag_shift=eps, precision=prec)
    x = delta.cpu().numpy()
    A = S + eps * np.eye(p.size)
    n = max(p.size, Ns)
    # the sample-space form subtracts vectors of size ||F|| / eps
    size = np.linalg.norm(A) * (np.linalg.norm(x) + (np.linalg.norm(F) / eps if solver != "cholesky" else 0.0))
    assert np.linalg.norm(A @ x - F) <= 8 * n * 2.0 ** -53 * (size + np.linalg.norm(F))


@pytest.mark.parametrize("bad", [np.nan, np.inf])
@pytest.mark.parametrize("at", [7, 40, 62])
def test_a_block_without_a_factor(ctx, bad, at):
    """A bias or weight of a hidden unit that is not a number reaches S through the
    unit's activations: the diagonal block leaves the fixed-point range and is done in
    FP64, where it spreads as it does in any Cholesky factorisation."""
    N, M, Ns = 7, 7, 65
    p, s, _, F = _system(N, M, Ns)
    p[at] = bad
    if np.isinf(bad):  # an infinite weight: infinity - infinity somewhere
        p[N + M:N + M + N] = bad
    delta = torch.empty(p.size, dtype=torch.float64, device=dev())
    nk.nk_sr_solve(ctx, cu(p), N, M, cu(s), cu(F), delta, solver="cholesky", diag_shift=0.01)
    assert torch.isnan(delta).all()
