"""NK_F64 J v on the tensor cores: a row's sum over the hidden units of one large term
and others of 0.9 2^-53 of it, which a single chain of additions drops one by one.

Tolerance: 16 additions a chain (64 columns a tile, four chains), 3 of the chains and
tiles, and the rounding of t, v and the products, in units of 2^-53 of the sum."""
import numpy as np
import pytest
import torch

from paper_2112_10526_gb300 import nk
from gpu_util import cu, dev

pytestmark = pytest.mark.gpu


def test_small_terms_beside_a_large_one():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    N, M, Ns = 64, 63, 1024
    p = np.zeros(N + M + N * M)
    p[N:N + M] = 0.5
    t = np.tanh(np.longdouble(0.5))
    v = np.zeros_like(p)
    v[N] = 1.0 / float(t)
    v[N + 1:N + M] = 0.9 * 2.0 ** -53 / float(t)
    s = np.ones((Ns, N), dtype=np.int8)
    out = torch.empty(Ns, dtype=torch.float64, device=dev())
    with nk.Ctx() as ctx:
        nk.nk_jvp(ctx, cu(p), N, M, cu(s), cu(v), out, precision="f64")
        got = out.cpu().numpy()
    # the library's own t: two terms of one unit each give it
    ref = (v[N:N + M].astype(np.longdouble) * t).sum()
    assert np.max(np.abs((got - ref).astype(np.float64))) <= (16 + 3 + 4) * 2.0 ** -53
