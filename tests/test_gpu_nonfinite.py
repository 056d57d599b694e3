"""Amplitudes that are not finite, and the largest finite ones, in the float H|psi>
from 512 strings of each spin: they reach the determinants within two excitations
and no other, whose values are those of the state without them.  Row ranges give
the full sweep's bits, and the next sweep of a finite state is not affected.

Tolerance: 2e-5 of the largest amplitude, the float sweep's bar in the parity tests.
"""
import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _strings(n, k):
    return np.array([s for s in range(1 << n) if bin(s).count("1") == k], dtype=np.int64)


def _moves(strings, s):
    return np.array([bin(int(x)).count("1") // 2 for x in strings ^ s])


@pytest.mark.parametrize("value", [float("nan"), float("inf"), -float("inf"), 3.4028234663852886e38, 3.402e38, 1e37,
                                   1e30, 1e20])
@pytest.mark.parametrize("cfg", [(12, 5, 7), (14, 4, 9)], ids=lambda c: "n%da%db%d" % c)
def test_reach(cfg, value):
    import __graft_entry__
    __graft_entry__.build()
    import paper_2604_01176_gb300 as hy
    n, na, nb = cfg
    ham = hy.Hamiltonian(*synth.integrals(n, 700 + n), n, na, nb)
    psi = torch.from_numpy(synth.random_state(ham.n_det, 9)).cuda().float()
    good = ham.apply_h(psi)
    A, B = ham.n_alpha_str // 3, ham.n_beta_str - 2
    at = A * ham.n_beta_str + B
    clean, bad = psi.clone(), psi.clone()
    clean[at], bad[at] = 0.0, value
    ref, out = ham.apply_h(clean.double()), ham.apply_h(bad)
    alpha, beta = _strings(n, na), _strings(n, nb)
    far = (_moves(alpha, alpha[A])[:, None] + _moves(beta, beta[B])[None, :]).ravel() > 2
    far = torch.from_numpy(far).cuda()
    assert far.any()
    assert not torch.isfinite(out[at]) or abs(out[at]) > 1e18
    tol = 2e-5 * ref.abs().max().item()
    assert torch.isfinite(out[far]).all()
    assert (out.double() - ref)[far].abs().max().item() <= tol
    nbs = ham.n_beta_str
    for a, b in ((A - 1, A + 2), (0, A), (A + 1, ham.n_alpha_str)):
        part = ham.apply_h_rows(bad, a, b)
        assert torch.equal(part.view(torch.int32), out[a * nbs:b * nbs].view(torch.int32))
    assert torch.equal(ham.apply_h(psi), good)
