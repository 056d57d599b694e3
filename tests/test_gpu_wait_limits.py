"""Waits of the tensor-core kernels at limits of a few polls: some run out and some
do not, in any role and at any stage.  The kernel ends either way, a timeout is
reported by the next call, a sweep without one has the usual bits, and the handle
works afterwards.
"""
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _run(cfg, limit):
    import __graft_entry__
    __graft_entry__.build()
    import paper_2604_01176_gb300 as hy
    n, na, nb = cfg
    ham = hy.Hamiltonian(*synth.integrals(n, 700 + n), n, na, nb)
    psi = torch.from_numpy(synth.random_state(ham.n_det, 9)).cuda().float()
    good = ham.apply_h(psi)
    for _ in range(3):
        ham.set_wait_limit(limit)
        out = ham.apply_h(psi)
        torch.cuda.synchronize()
        ham.set_wait_limit(1 << 26)
        try:
            again = ham.apply_h(psi)
        except hy.HyError as e:
            assert e.status == 4 and "timed out" in str(e)
        else:
            assert torch.equal(again, good) and torch.equal(out, good)
        assert torch.equal(ham.apply_h(psi), good)


# one tile and several, one J a block and many; 64 MMA rows in use (16 orbitals, 8 of a spin)
@pytest.mark.parametrize("limit", [1, 2, 5, 20, 100, 500])
@pytest.mark.parametrize("cfg", [(11, 1, 5), (11, 6, 5), (13, 7, 6), (16, 8, 2)],
                         ids=lambda c: "n%da%db%d" % c)
def test_wide_coupling(cfg, limit):
    _run(cfg, limit)


# the kernel of up to 10 orbitals: MMAs in flight at a timeout end before the block does
@pytest.mark.parametrize("limit", [1, 2, 5, 20, 100])
@pytest.mark.parametrize("cfg", [(6, 3, 3), (10, 5, 5), (10, 2, 7)], ids=lambda c: "n%da%db%d" % c)
def test_coupling(cfg, limit):
    _run(cfg, limit)
