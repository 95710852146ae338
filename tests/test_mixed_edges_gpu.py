"""NK_MIXED at the edges of its layouts: the register sweeps (a warp a chain for up
to four chunks of 128 units, two warps for up to 48; the last chunk ragged, and the
widths next to the ones they take), and the Jacobian products whose theta, tanh and FP32 pairs are one kernel
(units around its tiles of 64, rows around its tiles of 128).

Sweeps replay the oracle as the other sweep tests do, with their tie band, and equal
the general sweep's bit for bit (ln psi too, whose FP32 error grows without bound as
tanh(theta) nears 1).  The products are compared with numpy's FP64 ones: tanh(theta) enters as a pair of FP32
numbers (2^-47 of each value after both roundings) on the NK_MIXED side, so 1e-8 of
the largest entry leaves room for the cancellation of a few thousand terms."""
import numpy as np
import pytest
import torch

import oracle
from paper_2112_10526_gb300 import inputs as I
from paper_2112_10526_gb300 import nk
from gpu_util import cu, dev
from test_parity_gpu import _lnu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    with nk.Ctx() as c:
        yield c


@pytest.mark.parametrize("rule,N,edges", [("local", 37, None), ("exchange", 16, I.square_edges(4)),
                                          ("exchange", 36, I.square_edges(6))])
@pytest.mark.parametrize("M", [4, 8, 124, 128, 132, 256, 260, 508, 512, 516, 130, 2044, 2048, 2052, 3076, 4608, 6144])
def test_mixed_sweep_widths(ctx, rule, N, edges, M, nd=1, ns=3):
    C, sig = (37, 0.3) if M < 600 else (5, 0.05)
    p = I.rbm_params(N, M, 3 + M, sig)
    s0 = oracle.chain_init(N, C, rule, 9, 1)
    st, samples = cu(s0), torch.empty((C, ns, N), dtype=torch.int8, device=dev())
    lp = torch.empty((C, ns), dtype=torch.float64, device=dev())
    nacc = torch.zeros(C, dtype=torch.int64, device=dev())
    dec = torch.empty((C, nd + ns, N), dtype=torch.uint8, device=dev())
    e_dev = None if edges is None else cu(edges)
    nk.nk_metropolis_sweep(ctx, cu(p), N, M, rule, e_dev, st, 2, nd, ns, 9, 1, samples, lp, nacc, dec,
                           precision="mixed")
    got = dec.cpu().numpy()
    ref = oracle.metropolis(p, N, M, rule, edges, s0, 2, nd, ns, 9, 1, forced=got)
    two_d = _lnu(9, 1, C, N, nd + ns, 2) + np.where(ref["decisions"] == 1, 1, -1) * ref["margin"]
    allowed = ref["margin"] < 1e-4 * np.maximum(1.0, np.abs(two_d))
    assert not ((ref["decisions"] != got) & ~allowed).any()
    np.testing.assert_array_equal(samples.cpu().numpy(), ref["samples"])
    np.testing.assert_array_equal(st.cpu().numpy(), ref["state"])
    np.testing.assert_array_equal(nacc.cpu().numpy(), (got == 1).sum(axis=(1, 2)))
    # with units of zero weight up to a width that the general sweep takes, every
    # product, sum and renormalisation is the same
    Mw = 6160
    pw = np.zeros(N + Mw + Mw * N)
    pw[:N + M], pw[N + Mw:N + Mw + M * N] = p[:N + M], p[N + M:]
    outs = [cu(s0), torch.empty_like(samples), torch.empty_like(lp), torch.zeros_like(nacc), torch.empty_like(dec)]
    nk.nk_metropolis_sweep(ctx, cu(pw), N, Mw, rule, e_dev, outs[0], 2, nd, ns, 9, 1, *outs[1:], precision="mixed")
    for a, b in zip(outs, (st, samples, lp, nacc, dec)):
        assert M % 4 or torch.equal(a, b)  # other widths take their units in another order
    # without decisions and ln psi: the same chains
    st2, samples2 = cu(s0), torch.empty_like(samples)
    nk.nk_metropolis_sweep(ctx, cu(p), N, M, rule, e_dev, st2, 2, nd, ns, 9, 1, samples2, precision="mixed")
    assert torch.equal(st2, st) and torch.equal(samples2, samples)


@pytest.mark.parametrize("N", [5, 100])
@pytest.mark.parametrize("M", [1, 63, 64, 65, 200])
@pytest.mark.parametrize("Ns", [1, 129, 1300])
def test_mixed_jacobian_products(ctx, N, M, Ns):
    p, s = I.rbm_params(N, M, 7 + M, 0.2), I.random_configs(Ns, N, 5)
    rng = np.random.default_rng(1)
    g, v = rng.normal(size=Ns), rng.normal(size=N + M + N * M)
    sd = s.astype(np.float64)
    t = np.tanh(p[N:N + M] + sd @ p[N + M:].reshape(M, N).T)
    J = np.concatenate([sd, t, (t[:, :, None] * sd[:, None, :]).reshape(Ns, -1)], axis=1)
    dp, ds = cu(p), cu(s)
    out = torch.empty(v.size, dtype=torch.float64, device=dev())
    nk.nk_vjp(ctx, dp, N, M, ds, cu(g), out, precision="mixed")
    assert np.abs(out.cpu().numpy() - g @ J).max() < 1e-8 * np.abs(g).sum()
    jv = torch.empty(Ns, dtype=torch.float64, device=dev())
    nk.nk_jvp(ctx, dp, N, M, ds, cu(v), jv, precision="mixed")
    assert np.abs(jv.cpu().numpy() - J @ v).max() < 1e-8 * np.abs(v).sum()
    dJ = J - J.mean(axis=0)
    nk.nk_qgt_matvec(ctx, cu(v), out, 0.01, params=dp, N=N, M=M, s=ds, precision="mixed")
    ref = dJ.T @ (dJ @ v) / Ns + 0.01 * v
    assert np.abs(out.cpu().numpy() - ref).max() < 1e-8 * np.abs(v).sum()
