"""NK_F64 ln psi, J v, J^T g and the log-derivatives on both sides of the size
from which they run as 7-slice tensor-core products (f64_on_tensor: N M B >=
4e6), at ragged sizes, against plain FP64; and the FP64 semantics of
infinities, NaNs and extreme magnitudes on both routes.

Tolerance: an output is a sum of K products a_k b_k; recursive FP64 summation
errs by at most K 2^-53 sum |a_k b_k| on either side, the slices by K 2^-55
max |a_k b_k| <= K 2^-55 sum |a_k b_k|; the second factor of J v adds a few
units.  (2 K + 16) 2^-53 sum |a_k b_k| covers all of them.  J v and J^T g are
compared given the library's own tanh(theta) (the log-derivatives in the hidden
biases), which is itself checked against plain FP64 with the error of theta."""
import numpy as np
import pytest
import torch

from paper_2112_10526_gb300 import inputs as I
from paper_2112_10526_gb300 import nk
from gpu_util import cu, dev

pytestmark = pytest.mark.gpu

# (N, M, B): one tile and less, ragged tiles, just below and above 4e6, well above,
# more tiles than SMs (clusters; an odd count of row tiles), N beyond one resident row
SIZES = [(1, 1, 1), (16, 16, 256), (15, 17, 33), (37, 45, 1025), (50, 80, 999), (50, 80, 1000), (129, 191, 257),
         (144, 288, 1500), (30, 700, 1600), (600, 100, 300), (65, 40, 5000)]


@pytest.fixture(scope="module")
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    with nk.Ctx() as c:
        yield c


def _products(ctx, p, N, M, s, v, g):
    B = s.shape[0]
    pd, sd = cu(p), cu(s)
    lp = torch.empty(B, dtype=torch.float64, device=dev())
    jv = torch.empty(B, dtype=torch.float64, device=dev())
    jg = torch.empty(p.size, dtype=torch.float64, device=dev())
    O = torch.empty((min(B, 8), p.size), dtype=torch.float64, device=dev())
    nk.nk_rbm_logpsi(ctx, pd, N, M, sd, lp)
    nk.nk_jvp(ctx, pd, N, M, sd, cu(v), jv)
    nk.nk_vjp(ctx, pd, N, M, sd, cu(g), jg)
    nk.nk_jacobian(ctx, pd, N, M, sd, True, 0, O.shape[0], O)
    torch.cuda.synchronize()
    assert nk.nk_ctx_error(ctx) == 0
    rows = torch.empty((B, p.size), dtype=torch.float64, device=dev())
    nk.nk_jacobian(ctx, pd, N, M, sd, False, 0, B, rows)
    T = rows[:, N:N + M].cpu().numpy()
    return [x.cpu().numpy() for x in (lp, jv, jg, O)], T


def _reference(p, N, M, s, v, g, T_got):
    """The same and, for each, the sum of the magnitudes added up."""
    sd = s.astype(np.float64)
    a, b, W = p[:N], p[N:N + M], p[N + M:].reshape(M, N)
    with np.errstate(all="ignore"):
        th = b + sd @ W.T
        T = np.tanh(th)
        th_mag = np.abs(b) + np.abs(W).sum(1)
        err, lim = np.abs(T_got - T), (2 * N + 16) * 2.0 ** -53 * (1.0 + th_mag)
        assert (np.isnan(T_got) == np.isnan(T)).all()
        assert ((err <= lim) | np.isnan(T) | np.isinf(th)).all()
        assert (T_got[np.isinf(th)] == T[np.isinf(th)]).all()
        T = T_got
        x = np.abs(th)
        lp = sd @ a + (x + np.log1p(np.exp(-2 * x)) - np.log(2.0)).sum(1)
        lp_mag = np.abs(a).sum() + (np.abs(b) + np.abs(W).sum(1)).sum() + M
        va, vb, vW = v[:N], v[N:N + M], v[N + M:].reshape(M, N)
        jv = sd @ va + (T * (vb + sd @ vW.T)).sum(1)
        jv_mag = np.abs(va).sum() + (np.abs(T) * (np.abs(vb) + np.abs(vW).sum(1))).sum(1)
        Tg, Ta = T * g[:, None], np.abs(T) * np.abs(g)[:, None]
        jg = np.concatenate([sd.T @ g, Tg.sum(0), (Tg.T @ sd).ravel()])
        jg_mag = np.concatenate([np.full(N, np.abs(g).sum()), Ta.sum(0), np.repeat(Ta.sum(0), N)])
        rows = np.concatenate([sd, T, (T[:, :, None] * sd[:, None, :]).reshape(len(s), -1)], 1)
        O = (rows - rows.mean(0))[:8]
    return (lp, jv, jg, O), (lp_mag, jv_mag, jg_mag, 1.0)


@pytest.mark.parametrize("N,M,B", SIZES)
def test_f64_products_match_plain_fp64(ctx, N, M, B):
    p = I.rbm_params(N, M, 3, 0.2)
    rng = np.random.default_rng(N + M + B)
    s = I.random_configs(B, N, 5)
    v, g = rng.normal(size=p.size), rng.normal(size=B) * 10.0 ** rng.integers(-6, 3, B)
    got, T = _products(ctx, p, N, M, s, v, g)
    ref, mag = _reference(p, N, M, s, v, g, T)
    K = max(N + M, B) + 1
    for x, r, m in zip(got, ref, mag):
        assert (np.abs(x - r) <= (2 * K + 16) * 2.0 ** -53 * m).all()


@pytest.mark.parametrize("N,M,B", [(37, 45, 130), (129, 191, 257)])
def test_f64_products_keep_nonfinite_and_extreme_values(ctx, N, M, B):
    """A NaN or an infinity in one hidden unit, one tangent row or one sample's
    g reaches the outputs that FP64 arithmetic gives it, and no others; huge
    and tiny magnitudes come out as in FP64."""
    p = I.rbm_params(N, M, 3, 0.2)
    rng = np.random.default_rng(1)
    s = I.random_configs(B, N, 5)
    v, g = rng.normal(size=p.size), rng.normal(size=B)
    p[N + M + 2 * N + 1] = np.inf          # theta_2 = +-inf, tanh = +-1
    p[N + M + 4 * N + 3] = np.nan          # theta_4 = nan
    v[N + M + 6 * N + 5] = 1e300           # a row of J v far above the others
    g[7] = 1e290
    got, T = _products(ctx, p, N, M, s, v, g)
    ref, mag = _reference(p, N, M, s, v, g, T)
    K = max(N + M, B) + 1
    for x, r, m in zip(got, ref, mag):
        assert (np.isnan(x) == np.isnan(r)).all()
        assert (np.isinf(x) == np.isinf(r)).all()
        ok = np.isfinite(r)
        with np.errstate(all="ignore"):
            err, lim = np.abs(x - r), (2 * K + 16) * 2.0 ** -53 * np.broadcast_to(m, r.shape)
        assert (err[ok] <= np.where(np.isfinite(lim[ok]), lim[ok], np.inf)).all()
