"""The symmetric Jacobian's integer sums at the sizes where their layout changes:
one, two and four samples a block and a last block that is not full, one group
element, more outputs than threads, activations from 1e-9 to 1 side by side, and
configurations that are not +-1 (summed in FP64).

The activations are the library's own (G = 1 returns each as it is) and within
1e-12 of numpy's.
A term is rounded to half of 2^(ceil(log2 G) - 62) of a power of two at most twice
the feature's largest |t|, so to 2 G 2^-62 max|t|; G of them are summed exactly and
the result is rounded to FP64."""
import numpy as np
import pytest
import torch

from paper_2112_10526_gb300 import inputs as I
from paper_2112_10526_gb300 import nk
from gpu_util import cu, dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    with nk.Ctx() as c:
        yield c


def _run(ctx, N, alpha, perms, sigma, s):
    G, Ns = perms.shape[0], s.shape[0]
    rng = np.random.default_rng(N + alpha)
    p = rng.normal(size=1 + alpha * (1 + N))
    for f in range(alpha):  # each feature on its own scale
        sc = sigma * 10.0 ** (-3 * (f % 4))
        p[1 + f] *= sc
        p[1 + alpha + f * N:1 + alpha + (f + 1) * N] *= sc
    p, d_perms, ds = cu(p), cu(perms.astype(np.int32)), cu(s)
    M = alpha * G
    plain = torch.empty(N + M + M * N, dtype=torch.float64, device=dev())
    nk.nk_symm_expand(ctx, p, N, alpha, d_perms, plain)
    # every unit as a feature of its own under the trivial group: O_b is its t
    one = torch.cat([plain[:1], plain[N:]])
    J = torch.empty((Ns, one.numel()), dtype=torch.float64, device=dev())
    nk.nk_symm_jacobian(ctx, one, N, M, cu(np.arange(N, dtype=np.int32)[None]), ds, J)
    t = J[:, 1:1 + M].cpu().numpy()
    pl = plain.cpu().numpy()
    ref = np.tanh(pl[N:N + M] + s.astype(np.float64) @ pl[N + M:].reshape(M, N).T)
    assert np.abs(t - ref).max() < 1e-12
    t = t.reshape(Ns, alpha, G)
    O = torch.empty((Ns, 1 + alpha + alpha * N), dtype=torch.float64, device=dev())
    nk.nk_symm_jacobian(ctx, p, N, alpha, d_perms, ds, O)
    return t, O.cpu().numpy()


def _check(t, O, N, perms, s, per_term):
    assert np.isfinite(O).all()
    pick = np.unique(np.concatenate([np.arange(min(8, len(s))), np.arange(max(0, len(s) - 8), len(s))]))
    t, O, s = t[pick], O[pick], s[pick]
    Ns, alpha, G = t.shape
    tl, sl = t.astype(np.longdouble), s.astype(np.longdouble)
    big = np.abs(t).max(axis=2)  # [Ns, alpha]
    np.testing.assert_array_equal(O[:, 0], s.astype(np.float64).sum(axis=1))
    tol = per_term * G * big
    ref_b = tl.sum(axis=2)
    assert (np.abs(O[:, 1:1 + alpha] - ref_b) <= tol + 2.0 ** -52 * np.abs(ref_b)).all()
    ref_w = np.einsum("kfg,kgj->kfj", tl, sl[:, perms])
    W = O[:, 1 + alpha:].reshape(Ns, alpha, N)
    assert (np.abs(W - ref_w) <= tol[:, :, None] + 2.0 ** -52 * np.abs(ref_w)).all()


@pytest.mark.parametrize("perms", ["identity", "chain5", "chain33", "square8"])
@pytest.mark.parametrize("alpha", [1, 5, 17])
@pytest.mark.parametrize("Ns", [1, 607, 609, 1217, 1219])
def test_sums_over_the_group(ctx, perms, alpha, Ns):
    perms = {"identity": lambda: np.arange(6)[None], "chain5": lambda: I.translations_chain(5),
             "chain33": lambda: I.translations_chain(33), "square8": lambda: I.translations_square(8)}[perms]()
    G, N = perms.shape
    s = I.random_configs(Ns, N, 3)
    t, O = _run(ctx, N, alpha, perms, 0.3, s)
    _check(t, O, N, perms, s, 2.0 * G * 2.0 ** -62)


def test_configurations_that_are_not_plus_minus_one(ctx, Ns=1300, N=12, alpha=3):
    perms = I.translations_chain(N)
    s = I.random_configs(Ns, N, 3)
    s[5, 2], s[1297, 7], s[1299, 0] = 0, 3, -2
    t, O = _run(ctx, N, alpha, perms, 0.3, s)
    # FP64 sums of G terms at most 3 max|t|: G partial sums, each rounded to 2^-53
    _check(t, O, N, perms, s, 3 * N * 2.0 ** -53)
