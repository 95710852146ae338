"""Complex local energies with weights and activations beyond the range of the
exponentials that the flip ratios are products of: against ratios of cosh by the
oracle's logarithms (the tolerance of the other complex tests, 1e-10 of the batch's
rms)."""
import numpy as np
import pytest
import torch

from oracle import holo
from paper_2112_10526_gb300 import inputs as I
from paper_2112_10526_gb300 import nk
from gpu_util import cu, dev, ham_to_device

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    with nk.Ctx() as c:
        yield c


def _eloc(ctx, p, N, M, ham, s):
    h, _edges = ham_to_device(ham)
    e = torch.empty(len(s), dtype=torch.complex128, device=dev())
    nk.nk_crbm_local_energy(ctx, cu(p), N, M, h, cu(s), e)
    return e.cpu().numpy()


@pytest.mark.parametrize("kind", ["tfim", "heis"])
@pytest.mark.parametrize("M", [1, 33])
@pytest.mark.parametrize("w", [80.0, 90.0, 250.0, 400.0, 1e4])
def test_large_weights(ctx, kind, M, w):
    """One unit of weights +-w (+ a small rest), so that flips of one site, or of a
    pair, change |Re theta| by up to 4 w; the batch holds both sides."""
    N = 6
    ham = I.tfim_chain(N, -0.7, 1.1) if kind == "tfim" else I.heis_chain(N)
    p = I.complex_rbm_params(N, M, 5, 0.05)
    W = p[N + M:].reshape(M, N)
    W[M // 2, 0] += w
    W[M // 2, 1] -= w
    s = I.random_configs(40, N, 3, sz0=kind == "heis")
    ref = holo.local_energy(p, N, M, ham, s)
    ok = np.abs(ref) < 1e280  # the others overflow in the oracle as well
    assert ok.any()
    got = _eloc(ctx, p, N, M, ham, s)
    err = np.abs(got[ok] - ref[ok]) / np.maximum(np.abs(ref[ok]), 1.0)
    # ln cosh of |theta| <= 4 w is rounded to 4 w 2^-53
    assert np.max(err) <= 1e-10 + 16 * w * 2.0 ** -53


@pytest.mark.parametrize("b", [290.0, 310.0, 372.0, 380.0])
def test_large_activations(ctx, b):
    """theta near 2 W (beyond 372 its e^{-2 theta} is no longer a normal number): the
    flip back to small activations is the small ratio of the two."""
    N, M = 4, 3
    ham = I.tfim_chain(N, 0.0, 1.0)
    p = I.complex_rbm_params(N, M, 5, 0.05)
    p[N + 1] = b
    p[N + M:].reshape(M, N)[1, :2] = [b / 2, 0.3]
    s = np.array([[1, 1, 1, 1], [-1, 1, -1, 1], [-1, -1, 1, 1]], dtype=np.int8)
    ref = holo.local_energy(p, N, M, ham, s)
    got = _eloc(ctx, p, N, M, ham, s)
    err = np.abs(got - ref) / np.maximum(np.abs(ref), 1.0)
    assert np.max(err) <= 1e-10 + 16 * b * 2.0 ** -53


def test_a_nan_parameter(ctx):
    N, M = 6, 5
    p = I.complex_rbm_params(N, M, 5, 0.05)
    p[N + 2] = np.nan
    s = I.random_configs(8, N, 3)
    assert np.isnan(_eloc(ctx, p, N, M, I.tfim_chain(N, 1.0, 1.0), s).real).all()
