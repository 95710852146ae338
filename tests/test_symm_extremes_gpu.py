"""The symmetric Jacobian where its sums over the group run in FP64: more than 512
group elements, and activations at the lower end of the FP64 range."""
import numpy as np
import pytest
import torch

from paper_2112_10526_gb300 import nk
from gpu_util import cu, dev

pytestmark = pytest.mark.gpu


def _jacobian(p, N, alpha, perms, s):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    O = torch.empty((len(s), 1 + alpha + alpha * N), dtype=torch.float64, device=dev())
    with nk.Ctx() as ctx:
        nk.nk_symm_jacobian(ctx, cu(p), N, alpha, cu(perms.astype(np.int32)), cu(s), O)
        return O.cpu().numpy()


@pytest.mark.parametrize("G", [513, 8192])
def test_many_group_elements(G):
    """Two sites; the identity G - 1 times and the exchange last: activations of 1e-8,
    and one of 0.96.  Sums in group order: every partial sum is rounded to 2^-53, and
    each activation is within 2^-52 of itself and of the rounding of its theta, 2^-53."""
    w = np.array([0.3, 1.3 - 1e-8])  # theta = 1 + s_0 w_0 + s_1 w_1
    p = np.array([0.0, 1.0, *w])
    perms = np.tile(np.array([[0, 1]]), (G, 1))
    perms[-1] = [1, 0]
    s = np.array([[1, -1], [-1, 1]], dtype=np.int8)
    O = _jacobian(p, 2, 1, perms, s)
    LD = np.longdouble
    for k in range(2):
        sk = s[k][perms].astype(LD)  # [G, 2]
        th = LD(1.0) + sk @ w.astype(LD)
        t = np.tanh(th)
        slack = (2.0 ** -52 * np.abs(t) + 3 * 2.0 ** -53).sum()
        for got, terms in [(O[k, 1], t), (O[k, 2], t * sk[:, 0]), (O[k, 3], t * sk[:, 1])]:
            part = np.cumsum(terms)
            # theta's own rounding is the same for the equal terms: taken out by their value
            e1 = float((LD(got) - part[-1]))
            assert abs(e1) <= float(np.abs(part).sum()) * 2.0 ** -53 + float(slack)


def test_the_sums_are_of_the_activations_in_fp64():
    """The same, against the library's own activations (trivial group): the sum of the
    G rounded numbers, off by the roundings of the partial sums alone."""
    G = 8192
    w = np.array([0.3, 1.3 - 1e-8])
    s = np.array([[1, -1]], dtype=np.int8)
    one = np.array([0.0, 1.0, 1.0, w[0], w[1], w[1], w[0]])  # both orders as features of their own
    t = _jacobian(one, 2, 2, np.array([[0, 1]]), s)[0, 1:3].astype(np.longdouble)
    assert t[0] < 1e-7 and t[1] > 0.9
    perms = np.tile(np.array([[0, 1]]), (G, 1))
    perms[-1] = [1, 0]
    O = _jacobian(np.array([0.0, 1.0, *w]), 2, 1, perms, s)[0]
    terms = np.concatenate([np.full(G - 1, t[0]), [t[1]]])
    sg = np.concatenate([np.full(G - 1, 1.0), [-1.0]]).astype(np.longdouble)  # s_0 under the permutation
    for got, x in [(O[1], terms), (O[2], terms * sg), (O[3], -terms * sg)]:
        part = np.cumsum(x)
        assert abs(float(np.longdouble(got) - part[-1])) <= float(np.abs(part).sum()) * 2.0 ** -53


@pytest.mark.parametrize("size", [1e-280, 1e-290, 1e-300, 4e-308])
def test_tiny_activations(size):
    """All activations of one feature near the end of the normal numbers, the other's of
    ordinary size: relative accuracy of FP64 sums of five terms of one sign."""
    N, perms = 5, np.array([np.roll(np.arange(5), k) for k in range(5)])
    p = np.zeros(1 + 2 * (1 + N))
    p[1], p[2] = size, 0.3
    s = np.array([[1, -1, 1, 1, -1]] * 700, dtype=np.int8)
    O = _jacobian(p, N, 2, perms, s)
    np.testing.assert_allclose(O[:, 1], 5 * size, rtol=5 * 2.0 ** -52)
    np.testing.assert_allclose(O[:, 3:3 + N], size, rtol=8 * 2.0 ** -52)  # the spins sum to 1
    np.testing.assert_allclose(O[:, 2], 5 * np.tanh(0.3), rtol=8 * 2.0 ** -52)
