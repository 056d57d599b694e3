"""hy_energy without sigma as a handle's first call: sigma is formed in the workspace,
which has to have its full size before sigma's place in it is taken.  Tolerances:
1e-12 of the energy's scale in double, 1e-5 in float, the parity tests' bars.
"""
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
@pytest.mark.parametrize("cfg", [(2, 1, 1), (6, 3, 3), (10, 5, 5), (12, 5, 7), (14, 3, 7)],
                         ids=lambda c: "n%da%db%d" % c)
def test_energy_alone(cfg, dtype):
    import __graft_entry__
    __graft_entry__.build()
    import paper_2604_01176_gb300 as hy
    n, na, nb = cfg
    args = (*synth.integrals(n, 80 + n), n, na, nb)
    ref = hy.Hamiltonian(*args)
    psi = torch.from_numpy(synth.random_state(ref.n_det, 1)).cuda()
    sigma = ref.apply_h(psi)
    want = (psi @ sigma).item()
    scale = max(1.0, sigma.norm().item())
    tol = 1e-12 if dtype == torch.float64 else 1e-5
    ham = hy.Hamiltonian(*args)
    x = psi.to(dtype)
    assert abs(ham.energy(x).item() - want) <= tol * scale
    assert abs(ham.energy(x).item() - want) <= tol * scale
    other = torch.float32 if dtype == torch.float64 else torch.float64
    assert abs(ham.energy(psi.to(other)).item() - want) <= 1e-5 * scale
    assert abs(ham.energy(x).item() - want) <= tol * scale
