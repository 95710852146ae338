"""tanh(theta) of NK_F64 (the integer tanh of csrc/tanh64.cuh) on the GPU against
extended precision: W = 0, so that theta = b, read back as the log-derivatives
in the hidden biases.  0.53 units in the last place: half a unit of the final
rounding plus the few units of 2^-62 of the steps before it."""
import numpy as np
import pytest
import torch

from paper_2112_10526_gb300 import nk
from gpu_util import cu, dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("part", ["uniform", "log", "knots", "ends"])
def test_tanh_to_half_a_unit(part):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    M, rng = 8192, np.random.default_rng(3)
    if part == "uniform":
        b = rng.uniform(-20, 20, M)
    elif part == "log":
        b = 2.0 ** rng.uniform(-40, 5, M) * rng.choice([-1, 1], M)
    elif part == "knots":  # around k / 32: the table's points and the ties between them
        b = np.repeat(np.arange(1, M // 8 + 1) / 32.0, 8)[:M]
        for j in range(1, 4):
            b[j::8] = np.nextafter(b[j - 1::8], np.inf)
        for j in range(5, 8):
            b[j::8] = np.nextafter(b[j - 1::8], -np.inf)
    else:
        b = rng.uniform(18.5, 19.2, M)
        b[:12] = [0.0, -0.0, 5e-324, -1e-310, 1e-300, 2.0 ** -28, -(2.0 ** -28), 19.0625, 700.0, -1e308, np.inf, -np.inf]
        b[12] = np.nan
    p = np.concatenate([np.zeros(1), b, np.zeros(M)])
    s = np.ones((1, 1), dtype=np.int8)
    O = torch.empty((1, p.size), dtype=torch.float64, device=dev())
    with nk.Ctx() as c:
        nk.nk_jacobian(c, cu(p), 1, M, cu(s), False, 0, 1, O)
        torch.cuda.synchronize()
        got = O.cpu().numpy()[0, 1:1 + M]
    ref = np.tanh(b.astype(np.longdouble))
    assert (np.isnan(got) == np.isnan(b)).all()
    ok = ~np.isnan(b)
    ulp = np.spacing(np.abs(ref[ok]).astype(np.float64)).astype(np.longdouble)
    one = np.abs(ref[ok]).astype(np.float64) == 1.0
    assert (np.abs(got[ok] - ref[ok])[~one] <= 0.53 * ulp[~one]).all()
    assert (np.abs(got[ok])[one] == 1.0).all()
    assert (np.signbit(got[ok]) == np.signbit(0.0 + b[ok])).all()  # theta = 0 + b: -0 becomes +0
