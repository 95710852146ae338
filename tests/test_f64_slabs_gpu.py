"""NK_F64 ln psi and local energies of batches whose activations are taken a part at a
time: the bits of the parts by themselves, and a workspace that does not grow with the
batch."""
import pytest
import torch

from paper_2112_10526_gb300 import inputs as I
from paper_2112_10526_gb300 import nk
from gpu_util import cu, dev, ham_to_device

pytestmark = pytest.mark.gpu


def test_parts_and_workspace():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    N, M, Ns = 4, 8192, 20001  # 4096 samples a part; 1.3 GB of activations in all
    p, s = cu(I.rbm_params(N, M, 3, 0.05)), cu(I.random_configs(Ns, N, 5))
    h, _edges = ham_to_device(I.tfim_chain(N, 1.0, 1.0))

    def both(ctx, x, t=None):
        e, lp = (torch.empty(len(x), dtype=torch.float64, device=dev()) for _ in range(2))
        nk.nk_local_energy(ctx, p, N, M, h, x, e, t, precision="f64")
        nk.nk_rbm_logpsi(ctx, p, N, M, x, lp, precision="f64")
        return e, lp

    with nk.Ctx() as ctx:
        both(ctx, s[:16])
        torch.cuda.synchronize()
        free = torch.cuda.mem_get_info()[0]
        e, lp = both(ctx, s)
        torch.cuda.synchronize()
        assert free - torch.cuda.mem_get_info()[0] < 700 << 20
        t = torch.empty((5000, M), dtype=torch.float64, device=dev())
        e5, _ = both(ctx, s[:5000], t)
        assert torch.equal(e5, e[:5000])
        for k in range(0, Ns, 1500):
            x = s[k:k + 1500].contiguous()
            tk = torch.empty((len(x), M), dtype=torch.float64, device=dev())
            ek, lk = both(ctx, x, tk)
            assert torch.equal(ek, e[k:k + 1500]) and torch.equal(lk, lp[k:k + 1500])
            n = min(len(x), max(0, 5000 - k))
            assert torch.equal(tk[:n], t[k:k + n])
