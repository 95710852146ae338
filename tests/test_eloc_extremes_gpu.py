"""NK_F64 local energies of the Ising field where the flip ratios' factors 1 - s t tau
(t = tanh theta, tau = tanh 2 W) are at the ends of their range, against ratios of
cosh in extended precision.  M below and from 1024 on: the two mappings of the
kernel."""
import numpy as np
import pytest
import torch

from paper_2112_10526_gb300 import nk
from gpu_util import cu, dev

pytestmark = pytest.mark.gpu

LD = np.longdouble


@pytest.fixture(scope="module")
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    with nk.Ctx() as c:
        yield c


def _lncosh(x):
    x = np.abs(x)
    return x + np.log1p(np.exp(-2 * x)) - np.log(LD(2))


def _params(a, b, W):
    return np.concatenate([a, b, W.ravel()]).astype(np.float64)


def _field(ctx, a, b, W, s):
    """-sum_i psi(s with i flipped) / psi(s) per sample: the library's and the exact."""
    M, N = W.shape
    h = nk.make_ham("tfim", 0.0, 1.0, False, cu(np.array([[0, 1]], dtype=np.int32)))
    out = torch.empty(len(s), dtype=torch.float64, device=dev())
    nk.nk_local_energy(ctx, cu(_params(a, b, W)), N, M, h, cu(s), out, precision="f64")
    th = b.astype(LD) + s.astype(LD) @ W.T.astype(LD)
    ref = np.zeros(len(s), dtype=LD)
    for i in range(N):
        si = s[:, i].astype(LD)
        d = 2 * si[:, None] * W[:, i].astype(LD)[None, :]
        ref -= np.exp(-2 * a[i] * si + (_lncosh(th - d) - _lncosh(th)).sum(1))
    return out.cpu().numpy(), ref


@pytest.mark.parametrize("d", [25.0, 30.0, 40.0, 100.0])
@pytest.mark.parametrize("M,at", [(1, 0), (7, 2), (7, 6), (1030, 1), (1030, 1029)])
def test_saturated_units(ctx, M, at, d):
    """theta = 2 W = d of one unit: t = tau = 1 in FP64, factor 0, exact ratio 1 / cosh d
    (2.8e-11 at most); and t = 1, tau = -1, factor 2.  Tolerance: NK_F64's 1e-10."""
    N = 2
    g = np.random.default_rng(M)
    a, b, W = np.zeros(N), 0.01 * g.normal(size=M), 0.01 * g.normal(size=(M, N))
    b[at] = W[at, 0] = d / 2
    W[at, 1] = 0.0
    s = np.array([[1, 1], [1, -1]], dtype=np.int8)
    got, ref = _field(ctx, a, b, W, s)  # site 0: 1 / cosh d, site 1: about 1
    assert np.max(np.abs(got - ref)) <= 1e-10
    b[at] = -d * 1.5  # theta = -2 d, moved to -d for s_0 = -1: cosh d / cosh 2 d; from -d to -2 d for +1
    got, ref = _field(ctx, a, b, W, np.array([[1, 1], [-1, 1]], dtype=np.int8))
    assert abs(got[1] - ref[1]) <= 1e-10
    assert abs(got[0] / float(ref[0]) - 1) <= 1e-10


@pytest.mark.parametrize("d", [3.0, 5.0, 7.0, 9.0, 13.0, 15.0])
@pytest.mark.parametrize("M,units", [(2, [0, 1]), (5, [0, 1, 2, 3]), (9, [4, 5, 6, 7, 8]), (1030, [3, 35]),
                                     (1030, [64, 96, 128, 160])])
def test_several_small_factors(ctx, M, units, d):
    """Neighbouring factors of about 1 / cosh^2 d, which the product takes in pairs.

    Tolerance: t and tau are within 2^-53, so that a factor f errs by 2^-52 / f of
    itself; the product, the sum of logarithms K and the exponential by 2^-53 each per
    unit, of the logarithms' sizes: M (2 + d) 2^-53.  Both twice."""
    N = 2
    g = np.random.default_rng(M)
    a, b, W = 0.1 * g.normal(size=N), np.zeros(M), np.zeros((M, N))
    W[units] = 0.5 * d
    b[units] = 0.2 * g.normal(size=len(units))
    s = np.array([[1, 1], [1, -1], [-1, -1]], dtype=np.int8)
    got, ref = _field(ctx, a, b, W, s)
    th = b + s @ W.T
    f = [min(1 - abs(np.tanh(LD(th[k, j])) * np.tanh(2 * LD(W[j, 0]))) for j in units) for k in (0, 2)]
    for k, fk in zip((0, 2), f):
        tol = 2 * (len(units) * 2.0 ** -52 / float(fk) + M * (2 + d) * 2.0 ** -53)
        assert abs(float((LD(got[k]) - ref[k]) / ref[k])) <= tol


@pytest.mark.parametrize("M,at", [(1, 0), (33, 32), (1030, 5)])
@pytest.mark.parametrize("bad", ["bias", "weight"])
def test_a_nan_reaches_the_energy(ctx, M, at, bad):
    """A NaN among the parameters of a hidden unit makes every flip ratio NaN; a
    Heisenberg configuration without a pair to exchange has none to take part in."""
    N = 4
    g = np.random.default_rng(M)
    a, b, W = 0.1 * g.normal(size=N), 0.1 * g.normal(size=M), 0.1 * g.normal(size=(M, N))
    if bad == "bias":
        b[at] = np.nan
    else:
        W[at, 2] = np.nan
    s = np.array([[1, 1, 1, 1], [1, -1, 1, -1], [1, 1, -1, -1]], dtype=np.int8)
    edges = cu(np.array([[0, 1], [1, 2], [2, 3], [3, 0]], dtype=np.int32))
    p = cu(_params(a, b, W))
    out = torch.empty(len(s), dtype=torch.float64, device=dev())
    nk.nk_local_energy(ctx, p, N, M, nk.make_ham("tfim", 1.0, 1.0, False, edges), cu(s), out, precision="f64")
    assert torch.isnan(out).all()
    nk.nk_local_energy(ctx, p, N, M, nk.make_ham("heis", 1.0, 0.0, False, edges), cu(s), out, precision="f64")
    assert out.cpu().numpy()[0] == 4.0 and torch.isnan(out[1:]).all()
