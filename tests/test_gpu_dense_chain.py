"""Preparation and gradient of an ansatz on a small dense state in one launch
each, against the same chain by single calls: apply_excitation from the
Hartree-Fock state, apply_h, and per-operator gradients on the vectors walked
back.  Sizes: one and few determinants per CTA, ragged string counts, the
largest that fits (63,504), the first that does not (12, 2, 8: 32,670 fits;
11, 6, 5: 213,444 does not), empty ansatz, one and many operators.

Tolerances: the single calls use the same roundings per rotation, so states
agree to 1e-14 (double) and 1e-6 (float, whose squared norm is summed in another
order); energies and gradients to 1e-12 and 1e-5, the parity tests' bars.
"""
import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

CFGS = [(2, 1, 1, 1), (3, 2, 1, 3), (5, 1, 4, 6), (6, 3, 3, 0), (6, 3, 3, 40), (9, 2, 6, 7),
        (10, 5, 5, 13), (12, 2, 8, 5), (11, 6, 5, 4)]


@pytest.mark.parametrize("kind", ["sd", "qeb"])
@pytest.mark.parametrize("precision", ["f64", "mixed"])
@pytest.mark.parametrize("cfg", CFGS, ids=[f"n{n}a{a}b{b}L{k}" for n, a, b, k in CFGS])
def test_chain_matches_single_calls(cfg, precision, kind):
    import __graft_entry__
    __graft_entry__.build()
    import paper_2604_01176_gb300 as hy
    n, na, nb, length = cfg
    ham = hy.Hamiltonian(*synth.integrals(n, 90 + n), n, na, nb)
    pool = hy.Pool(ham, kind)
    rng = np.random.default_rng(n + length)
    ops = rng.integers(0, len(pool), length)
    th = 0.3 * rng.standard_normal(length)
    dt = torch.float64 if precision == "f64" else torch.float32
    ad = hy.Adapt(ham, pool, precision, max_iter=max(length, 1))
    ad.set_ansatz(ops, th)
    e, g = ad.evaluate(th, dt)
    psi = ham.hf_state(dt)
    n2 = torch.ones((), dtype=torch.float64, device="cuda")
    for k, t in zip(ops, th):
        if dt == torch.float32:
            pool.apply_excitation_tracked(int(k), float(t), psi, n2)
        else:
            pool.apply_excitation(int(k), float(t), psi)
    if dt == torch.float32 and length:
        ham.renormalize(psi, n2)
    f64 = dt == torch.float64
    assert torch.max(torch.abs(ad.state(dt) - psi)).item() <= (1e-14 if f64 else 1e-6)
    sigma = ham.apply_h(psi)
    tol = 1e-12 if f64 else 1e-5
    scale = max(1.0, sigma.abs().max().item() * 4)
    assert abs(e - ham.energy(psi, sigma).item()) <= tol * scale
    phi, lam = psi.clone(), sigma.clone()
    ref = np.zeros(length)
    for l in range(length - 1, -1, -1):
        one = torch.tensor([ops[l]], dtype=torch.int32, device="cuda")
        ref[l] = pool.gradients(phi, lam, ops=one).item()
        pool.apply_excitation(int(ops[l]), -float(th[l]), phi)
        pool.apply_excitation(int(ops[l]), -float(th[l]), lam)
    assert np.abs(g - ref).max(initial=0.0) <= tol * scale


@pytest.mark.parametrize("precision", ["f64", "mixed"])
@pytest.mark.parametrize("cfg", [(6, 3, 3), (8, 4, 4), (10, 5, 5)], ids=lambda c: "n%da%db%d" % c)
def test_longest_ansatz_of_one_launch(cfg, precision):
    """192 operators are walked in one launch each way (its largest shared memory), 193 by
    the per-rotation launches; a last operator at angle 0 changes neither the energy
    nor the other derivatives."""
    import __graft_entry__
    __graft_entry__.build()
    import paper_2604_01176_gb300 as hy
    n, na, nb = cfg
    ham = hy.Hamiltonian(*synth.integrals(n, 90 + n), n, na, nb)
    pool = hy.Pool(ham)
    rng = np.random.default_rng(n)
    ops = rng.integers(0, len(pool), 193)
    th = np.append(0.1 * rng.standard_normal(192), 0.0)
    dt = torch.float64 if precision == "f64" else torch.float32
    ad = hy.Adapt(ham, pool, precision, max_iter=193)
    got = []
    for length in (192, 193):
        ad.set_ansatz(ops[:length], th[:length])
        got.append(ad.evaluate(th[:length], dt))
    (e1, g1), (e2, g2) = got
    tol = 1e-12 if precision == "f64" else 1e-5
    scale = max(1.0, abs(e1))
    assert abs(e1 - e2) <= tol * scale
    assert np.abs(g1 - g2[:192]).max() <= tol * scale
