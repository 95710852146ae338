"""NK_F64 sweeps against the oracle where their FP32 screening is hardest: one
hidden unit to several hundred, ragged widths, weights small (every proposal
near the threshold of its bound) and large (ratio factors near 0 and 2, which
only FP64 can judge), all three rules.

The oracle follows the GPU's decisions and recomputes its own; they may differ
only where |2 dlnpsi - ln u| < 1e-9, the rounding of either side (the tolerance
of the other sweep tests).  ln psi is compared with numpy's log1p(2 sinh^2(x /
2)): the oracle's form loses the leading digits of ln cosh at sigma = 1e-6."""
import numpy as np
import pytest
import torch

import oracle
from paper_2112_10526_gb300 import inputs as I
from paper_2112_10526_gb300 import nk
from gpu_util import cu, dev, rel_err

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    with nk.Ctx() as c:
        yield c


@pytest.mark.parametrize("rule,N,edges", [("local", 13, None), ("exchange", 16, I.square_edges(4)),
                                          ("hamiltonian", 16, I.square_edges(4))])
@pytest.mark.parametrize("M", [1, 31, 33, 64, 127, 129, 300])
@pytest.mark.parametrize("sig", [1e-6, 0.3, 3.0])
def test_f64_sweep_decisions_are_those_of_fp64(ctx, rule, N, edges, M, sig, C=33):
    nd, ns = 2, 3
    p = I.rbm_params(N, M, 7 + M, sig)
    s0 = oracle.chain_init(N, C, rule, 5, 2)
    st, samples = cu(s0), torch.empty((C, ns, N), dtype=torch.int8, device=dev())
    lp = torch.empty((C, ns), dtype=torch.float64, device=dev())
    nacc = torch.zeros(C, dtype=torch.int64, device=dev())
    dec = torch.empty((C, nd + ns, N), dtype=torch.uint8, device=dev())
    nk.nk_metropolis_sweep(ctx, cu(p), N, M, rule, None if edges is None else cu(edges), st, 3, nd, ns, 5, 2, samples,
                           lp, nacc, dec)
    got = dec.cpu().numpy()
    ref = oracle.metropolis(p, N, M, rule, edges, s0, 3, nd, ns, 5, 2, forced=got)
    assert not ((ref["decisions"] != got) & (ref["margin"] >= 1e-9)).any()
    np.testing.assert_array_equal(samples.cpu().numpy(), ref["samples"])
    np.testing.assert_array_equal(st.cpu().numpy(), ref["state"])
    np.testing.assert_array_equal(nacc.cpu().numpy(), (got == 1).sum(axis=(1, 2)))
    sd = ref["samples"].astype(np.float64)
    th = np.abs(p[N:N + M] + sd @ p[N + M:].reshape(M, N).T)
    lncosh = np.where(th < 1.0, np.log1p(2.0 * np.sinh(0.5 * np.minimum(th, 1.0)) ** 2),
                      th + np.log1p(np.exp(-2.0 * th)) - np.log(2.0))
    assert rel_err(lp.cpu().numpy(), sd @ p[:N] + lncosh.sum(-1)) < 1e-10


def test_f64_sweep_of_many_chains(ctx):
    """More chains than the speculative form takes (1216)."""
    test_f64_sweep_decisions_are_those_of_fp64(ctx, "exchange", 16, I.square_edges(4), 33, 0.3, C=1300)
