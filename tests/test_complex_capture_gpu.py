"""nk_crbm_local_energy uses no workspace: the first call of a context can be captured
into a CUDA graph, and two calls of one context can run at the same time on two
streams."""
import numpy as np
import pytest
import torch

from paper_2112_10526_gb300 import inputs as I
from paper_2112_10526_gb300 import nk
from gpu_util import cu, dev, ham_to_device

pytestmark = pytest.mark.gpu

N, M, NS = 20, 20, 512


def _case(seed):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    return cu(I.complex_rbm_params(N, M, seed, 0.1)), cu(I.random_configs(NS, N, seed))


def _ref(p, s, h):
    out = torch.empty(NS, dtype=torch.complex128, device=dev())
    with nk.Ctx() as c:
        nk.nk_crbm_local_energy(c, p, N, M, h, s, out)
        torch.cuda.synchronize()
    return out.cpu().numpy()


def test_first_call_in_a_graph():
    p, s = _case(3)
    h, _edges = ham_to_device(I.tfim_chain(N, -0.7, 1.1))
    ref = _ref(p, s, h)
    out = torch.zeros(NS, dtype=torch.complex128, device=dev())
    torch.cuda.synchronize()
    with nk.Ctx() as c:
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g):
            nk.nk_crbm_local_energy(c, p, N, M, h, s, out)
        for _ in range(3):
            out.zero_()
            g.replay()
            torch.cuda.synchronize()
            np.testing.assert_array_equal(out.cpu().numpy(), ref)
        del g


def test_two_streams_of_one_context():
    h, _edges = ham_to_device(I.tfim_chain(N, -0.7, 1.1))
    cases = [_case(k) for k in (3, 4)]
    refs = [_ref(p, s, h) for p, s in cases]
    streams = [torch.cuda.Stream() for _ in cases]
    outs = [torch.empty((20, NS), dtype=torch.complex128, device=dev()) for _ in cases]
    torch.cuda.synchronize()
    with nk.Ctx() as c:
        for r in range(20):
            for (p, s), st, out in zip(cases, streams, outs):
                nk.nk_crbm_local_energy(c, p, N, M, h, s, out[r], stream=st)
        torch.cuda.synchronize()
    for out, ref in zip(outs, refs):
        assert (out.cpu().numpy() == ref).all()
