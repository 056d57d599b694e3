"""Float H|psi> with the tensor-core coupling of 11 and more orbitals against
the FP32 SIMT coupling and the double sweep: one column tile and many, ragged
last tiles, one and nearly all orbitals occupied (tiles of one operand stage),
a full and an empty spin, row ranges; and its waits, which run out and are
reported when its MMAs are withheld.

Tolerance: 2e-5 of the largest amplitude, the float sweep's bar in the parity
tests.
"""
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

CFGS = [(11, 6, 5), (11, 2, 9), (11, 11, 5), (11, 5, 0), (12, 6, 6), (12, 3, 12), (12, 2, 1), (13, 7, 5),
        (14, 3, 13), (15, 1, 8), (16, 2, 7), (16, 3, 1)]


def _ham(cfg):
    import __graft_entry__
    __graft_entry__.build()
    import paper_2604_01176_gb300 as hy
    n, na, nb = cfg
    ham = hy.Hamiltonian(*synth.integrals(n, 400 + n), n, na, nb)
    psi = torch.from_numpy(synth.random_state(ham.n_det, 8)).cuda().float()
    return hy, ham, psi


@pytest.mark.parametrize("cfg", CFGS, ids=["n%da%db%d" % c for c in CFGS])
def test_wide_coupling_matches_simt_and_double(cfg):
    hy, ham, psi = _ham(cfg)
    ham.set_coupling("simt")
    simt = ham.apply_h(psi)
    ham.set_coupling("tensor")
    out = torch.full_like(psi, float("nan"))
    ham.apply_h(psi, out=out)
    ref = ham.apply_h(psi.double())
    scale = ref.abs().max().item()
    assert (out - simt).abs().max().item() <= 2e-5 * scale
    assert (out.double() - ref).abs().max().item() <= 2e-5 * scale
    again = ham.apply_h(psi)
    assert torch.equal(again, out)
    a = ham.n_alpha_str // 2
    assert torch.equal(ham.apply_h_rows(psi, a, ham.n_alpha_str), out[a * ham.n_beta_str:])


@pytest.mark.parametrize("cfg", [(11, 2, 1), (11, 3, 5), (12, 2, 3)])
def test_withheld_waits_run_out_and_are_reported(cfg):
    """No stage is ever released: the builders' waits give up after the short
    limit set here, every other role follows, the next call reports it and the
    handle then works."""
    hy, ham, psi = _ham(cfg)
    good = ham.apply_h(psi)
    ham.set_wait_limit(2000)
    ham.set_coupling("withheld")
    ham.apply_h(psi)
    torch.cuda.synchronize()
    with pytest.raises(hy.HyError) as ei:
        ham.apply_h(psi)
    assert ei.value.status == 4 and "timed out" in str(ei.value)
    ham.set_coupling("tensor")
    ham.set_wait_limit(1 << 26)
    assert torch.equal(ham.apply_h(psi), good)
