"""Double sparse evaluations beyond the support programs (sigma on the rows of a
support of more than 65,536 determinants) against the dense sweeps: runs of more
rows than a block has threads, short runs, one electron of a spin, every beta
string present and few.

Tolerances: energies 1e-10, gradients 1e-9, as for the other sparse evaluations.
"""
import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

CFGS = [(12, 3, 6), (12, 6, 3), (12, 6, 6), (16, 1, 8), (16, 8, 1), (13, 5, 4)]


@pytest.mark.parametrize("cfg", CFGS, ids=["n%da%db%d" % c for c in CFGS])
def test_support_rows_match_dense(cfg):
    import __graft_entry__
    __graft_entry__.build()
    import paper_2604_01176_gb300 as hy
    n, na, nb = cfg
    ham = hy.Hamiltonian(*synth.integrals(n, 900 + n), n, na, nb)
    pool = hy.Pool(ham)
    sp = hy.Adapt(ham, pool, "f64", max_iter=160, sparse=True, sparse_cap=ham.n_det)
    de = hy.Adapt(ham, pool, "f64", max_iter=160)
    rng = np.random.default_rng(17)
    for length in range(20, 161, 20):
        ops = [int(k) for k in rng.choice(len(pool), length)]
        th = rng.uniform(0.1, 0.7, length)
        de.set_ansatz(ops, th)
        de.evaluate(th, torch.float64)
        m = int((de.state(torch.float64) != 0).sum())
        if m > 65536:
            break
    assert m > 65536
    sp.set_ansatz(ops, th)
    sp.evaluate(th, torch.float64)                  # lists the support
    for t in (th, th + rng.normal(0, 0.1, length)):
        e, g = sp.evaluate(t, torch.float64)
        e_d, g_d = de.evaluate(t, torch.float64)
        assert abs(e - e_d) < 1e-10
        assert np.abs(np.asarray(g) - np.asarray(g_d)).max() < 1e-9
