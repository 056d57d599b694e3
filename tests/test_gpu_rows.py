"""Double-precision H psi by rows (one launch over rows x column chunks):
string counts at the edges of its chunks, slices and range, against sampled
Slater-Condon rows of the oracle, and a row range against the whole.

Tolerance: FP64 amplitudes 1e-12 max-abs, as in the parity tests.
"""
import numpy as np
import pytest

import oracle
import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

# one string per spin; one and two electrons; 64 / 65-column chunks' edges (66,
# 126 strings); many columns on few rows, sliced (13, 1, 6) and (12, 2, 6); just
# above the sliced sizes (11, 6, 5); 320-column chunks (13, 7, 6); many rows on
# few columns (16, 8, 2); beyond the range (14, 2, 6: 3,003 strings)
CFGS = [(1, 1, 0), (4, 4, 2), (12, 6, 1), (12, 1, 2), (9, 5, 4), (13, 1, 6), (12, 2, 6),
        (11, 6, 5), (13, 7, 6), (16, 8, 2), (14, 2, 6)]


@pytest.mark.parametrize("cfg", CFGS, ids=[f"n{n}a{a}b{b}" for n, a, b in CFGS])
def test_rows_match_oracle(cfg):
    import __graft_entry__
    __graft_entry__.build()
    import paper_2604_01176_gb300 as hy
    n, na, nb = cfg
    h1, h2, ec = synth.integrals(n, 300 + n)
    ham = hy.Hamiltonian(h1, h2, ec, n, na, nb)
    ref = oracle.System(h1, h2, ec, n, na, nb)
    x = synth.random_state(ham.n_det, 9)
    psi = torch.from_numpy(x).cuda()
    sigma = torch.full_like(psi, float("nan"))
    ham.apply_h(psi, out=sigma)
    rng = np.random.default_rng(n)
    rows = np.unique(np.concatenate([[0, ham.n_det - 1], rng.integers(0, ham.n_det, 400)]))
    got = sigma[torch.from_numpy(rows).cuda()].cpu().numpy()
    assert np.abs(got - ref.sigma_rows(x, rows)).max() < 1e-12
    assert bool(torch.isfinite(sigma).all())
    a, b = ham.n_alpha_str // 3, ham.n_alpha_str
    part = ham.apply_h_rows(psi, a, b)
    assert torch.equal(part, sigma[a * ham.n_beta_str:])
