"""The complex RBM's sampler and local energies at the edges of their warp
layout (hidden units around 32 and 64, more sites or edges than lanes) and with
weights from small to large, against the oracle: chains bit-exact (the FP32
screening may only hand over to FP64, never decide differently), local energies
to 1e-10 of the batch's rms (the tolerance of the other complex tests)."""
import numpy as np
import pytest
import torch

from oracle import holo
from paper_2112_10526_gb300 import inputs as I
from paper_2112_10526_gb300 import nk
from gpu_util import cu, dev, ham_to_device

pytestmark = pytest.mark.gpu

HAMS = {"tfim9": (9, lambda: I.tfim_chain(9, -0.7, 1.1), "local"),
        "heis4x4": (16, lambda: I.heis_square(4), "exchange"),
        "tfim40": (40, lambda: I.tfim_chain(40, 1.0, 0.6), "local"),
        "j1j2-6x6": (36, lambda: I.j1j2_square(6), "exchange")}


@pytest.fixture(scope="module")
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    with nk.Ctx() as c:
        yield c


@pytest.mark.parametrize("name", list(HAMS))
@pytest.mark.parametrize("M", [1, 31, 33, 70])
@pytest.mark.parametrize("sig", [0.01, 0.3, 1.0])
def test_complex_eloc_and_chains(ctx, name, M, sig):
    N, hf, rule = HAMS[name]
    ham = hf()
    p = I.complex_rbm_params(N, M, 11 + M, sig)
    s = I.random_configs(21, N, 3, sz0=rule == "exchange")
    h, edges = ham_to_device(ham)
    e = torch.empty(len(s), dtype=torch.complex128, device=dev())
    nk.nk_crbm_local_energy(ctx, cu(p), N, M, h, cu(s), e)
    ref = holo.local_energy(p, N, M, ham, s)
    assert np.max(np.abs(e.cpu().numpy() - ref)) <= 1e-10 * np.sqrt(np.mean(np.abs(ref) ** 2))
    C = 5
    sd, samples = cu(s[:C]), torch.empty((C, 2, N), dtype=torch.int8, device=dev())
    nacc = torch.zeros(C, dtype=torch.int64, device=dev())
    nk.nk_crbm_metropolis(ctx, cu(p), N, M, rule, None if rule == "local" else edges, sd, 2, 1, 2, 77, 1, samples, nacc)
    state, want = holo.metropolis(p, N, M, rule, ham["edges"], s[:C], 2, 1, 2, 77, 1)
    np.testing.assert_array_equal(samples.cpu().numpy(), want)
    np.testing.assert_array_equal(sd.cpu().numpy(), state)
