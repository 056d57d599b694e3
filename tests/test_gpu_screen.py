"""The whole-pool double-precision screen (summed by string pattern) against
the per-operator kernel that serves operator lists: pool.gradients(psi, sigma)
against the same pool passed as a list.  Sizes cover empty spins, one-string
spins, ragged string counts, odd groups of same-spin vectors and the three
staging configurations (n = 13, 15 and 16 are the largest of each).

Tolerance: both sum the same products in double; |g| <= 4 |sigma| |psi| = 4
here and each sum rounds at 2^-53 of its partial sums, so 1e-12 is far above
any reordering of up to 10^9 terms of random sign (~1e-15 expected).
"""
import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

CFGS = [(2, 1, 0), (2, 1, 1), (3, 3, 1), (4, 0, 2), (4, 3, 1), (5, 1, 4), (6, 3, 3), (7, 4, 3),
        (9, 2, 6), (11, 6, 5), (13, 7, 5), (13, 6, 7), (15, 8, 7), (16, 8, 8)]


@pytest.mark.parametrize("kind", ["sd", "qeb"])
@pytest.mark.parametrize("cfg", CFGS, ids=[f"n{n}a{a}b{b}" for n, a, b in CFGS])
def test_whole_pool_matches_operator_list(cfg, kind):
    import __graft_entry__
    __graft_entry__.build()
    import paper_2604_01176_gb300 as hy
    n, na, nb = cfg
    if n == 16 and kind == "qeb":
        pytest.skip("same staging configuration as the spin-adapted pool")
    ham = hy.Hamiltonian(*synth.integrals(n, 50 + n), n, na, nb)
    pool = hy.Pool(ham, kind)
    g = torch.Generator(device="cuda")
    g.manual_seed(n)
    v = torch.randn((2, ham.n_det), dtype=torch.float64, device="cuda", generator=g)
    psi, sigma = v[0] / v[0].norm(), v[1] / v[1].norm()
    every = torch.arange(len(pool), dtype=torch.int32, device="cuda")
    whole = torch.full((len(pool),), np.nan, dtype=torch.float64, device="cuda")
    pool.gradients(psi, sigma, out=whole)
    listed = pool.gradients(psi, sigma, ops=every)
    assert torch.max(torch.abs(whole - listed)).item() <= 1e-12


def test_packed_molecules_match_their_own_screens():
    """One launch over molecules of different staging sizes."""
    import __graft_entry__
    __graft_entry__.build()
    import paper_2604_01176_gb300 as hy
    sizes = [(6, 3, 3), (13, 6, 7), (4, 0, 2), (9, 5, 4), (14, 7, 7)]
    hams = [hy.Hamiltonian(*synth.integrals(n, 70 + i), n, a, b) for i, (n, a, b) in enumerate(sizes)]
    pools = [hy.Pool(h) for h in hams]
    batch = hy.Batch(hams)
    batch.set_pools(pools)
    psi = batch.pack([torch.from_numpy(synth.random_state(h.n_det, 1)).cuda() for h in hams])
    sigma = batch.pack([torch.from_numpy(synth.random_state(h.n_det, 2)).cuda() for h in hams])
    g = batch.gradients(psi, sigma)
    for m, (x, y) in enumerate(zip(batch.unpack(psi), batch.unpack(sigma))):
        lo, hi = batch.pool_offsets[m], batch.pool_offsets[m + 1]
        every = torch.arange(len(pools[m]), dtype=torch.int32, device="cuda")
        if len(every):
            ref = pools[m].gradients(x, y, ops=every)
            assert torch.max(torch.abs(g[lo:hi] - ref)).item() <= 1e-12


@pytest.mark.parametrize("kind", ["sd", "qeb"])
@pytest.mark.parametrize("cfg", CFGS[:9], ids=[f"n{n}a{a}b{b}" for n, a, b in CFGS[:9]])
def test_small_molecule_in_a_batch(cfg, kind):
    """Below 16,384 determinants a molecule alone is screened per operator; in a
    batch it takes the screen by pattern."""
    import __graft_entry__
    __graft_entry__.build()
    import paper_2604_01176_gb300 as hy
    n, na, nb = cfg
    ham = hy.Hamiltonian(*synth.integrals(n, 50 + n), n, na, nb)
    pool = hy.Pool(ham, kind)
    batch = hy.Batch([ham])
    batch.set_pools([pool])
    psi = torch.from_numpy(synth.random_state(ham.n_det, 3)).cuda()
    sigma = torch.from_numpy(synth.random_state(ham.n_det, 4)).cuda()
    whole = batch.gradients(batch.pack([psi]), batch.pack([sigma]))
    every = torch.arange(len(pool), dtype=torch.int32, device="cuda")
    listed = pool.gradients(psi, sigma, ops=every)
    assert torch.max(torch.abs(whole - listed)).item() <= 1e-12


@pytest.mark.parametrize("kind", ["sd", "qeb"])
@pytest.mark.parametrize("cfg", [(10, 5, 5), (11, 6, 5), (12, 9, 4), (13, 4, 9), (13, 7, 5), (14, 7, 7),
                                 (15, 8, 7), (16, 4, 8), (16, 8, 8)],
                         ids=lambda c: "n%da%db%d" % c)
def test_float_pool_keeps_the_operator_lists_sums(cfg, kind):
    """Float: the same float sums per thread as the per-operator kernel (same
    row chunks for a list of the whole pool), so only the double sums of 256
    threads differ: 1e-13 of them, |g| <= 4 on normalised vectors.  Sizes: one to
    fourteen table entries per thread and pattern, both stagings, several chunks
    (small pools), shares of patterns that do not divide."""
    import __graft_entry__
    __graft_entry__.build()
    import paper_2604_01176_gb300 as hy
    n, na, nb = cfg
    if n == 16 and (kind == "qeb") != (na == 4):
        pytest.skip("one pool per 16-orbital size")
    ham = hy.Hamiltonian(*synth.integrals(n, 50 + n), n, na, nb)
    pool = hy.Pool(ham, kind)
    g = torch.Generator(device="cuda")
    g.manual_seed(n + na)
    v = torch.randn((2, ham.n_det), dtype=torch.float32, device="cuda", generator=g)
    psi, sigma = v[0] / v[0].norm(), v[1] / v[1].norm()
    every = torch.arange(len(pool), dtype=torch.int32, device="cuda")
    whole = torch.full((len(pool),), np.nan, dtype=torch.float64, device="cuda")
    pool.gradients(psi, sigma, out=whole)
    listed = pool.gradients(psi, sigma, ops=every)
    assert torch.max(torch.abs(whole - listed)).item() <= 1e-13


@pytest.mark.parametrize("kind", ["sd", "qeb"])
@pytest.mark.parametrize("cfg", [(16, 1, 8), (16, 15, 8), (16, 8, 1), (16, 2, 8), (13, 11, 6), (12, 2, 6), (16, 3, 4),
                                 (15, 1, 9)], ids=lambda c: "n%da%db%d" % c)
def test_few_strings_of_a_spin(cfg, kind):
    """Few strings of one spin: the other's patterns are cut in slices as well (16,384
    determinants and more, so alone the pool takes the screen by pattern)."""
    import __graft_entry__
    __graft_entry__.build()
    import paper_2604_01176_gb300 as hy
    n, na, nb = cfg
    ham = hy.Hamiltonian(*synth.integrals(n, 50 + n), n, na, nb)
    assert ham.n_det >= 16384
    pool = hy.Pool(ham, kind)
    g = torch.Generator(device="cuda")
    g.manual_seed(n)
    v = torch.randn((2, ham.n_det), dtype=torch.float64, device="cuda", generator=g)
    psi, sigma = v[0] / v[0].norm(), v[1] / v[1].norm()
    every = torch.arange(len(pool), dtype=torch.int32, device="cuda")
    whole = torch.full((len(pool),), np.nan, dtype=torch.float64, device="cuda")
    pool.gradients(psi, sigma, out=whole)
    listed = pool.gradients(psi, sigma, ops=every)
    assert torch.max(torch.abs(whole - listed)).item() <= 1e-12
