"""Calls with little device memory left: scratch that does not fit is done without, and
nothing is held that is not used.  The rest of the device is filled by one tensor.
"""
import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

MB = 1 << 20


def _free():
    torch.cuda.synchronize()
    return torch.cuda.mem_get_info()[0]


def _leave(nbytes):
    """Fills the device up to about nbytes."""
    torch.cuda.empty_cache()
    return torch.empty(_free() - nbytes, dtype=torch.uint8, device="cuda")


def test_same_spin_operands_of_one_spin():
    """Room for the sweep's workspace and the operands of one spin (16 MB of alpha, 63 of
    beta): the workspace is had, neither spin's operands are kept, the values are right.
    Tolerance: 2e-5 of the largest amplitude, the float sweep's bar in the parity tests."""
    import __graft_entry__
    __graft_entry__.build()
    import paper_2604_01176_gb300 as hy
    n, na, nb = 14, 4, 9
    ham = hy.Hamiltonian(*synth.integrals(n, 714), n, na, nb)
    psi = torch.from_numpy(synth.random_state(ham.n_det, 9)).cuda()
    ref = ham.apply_h(psi)
    x, out = psi.float(), torch.empty_like(psi, dtype=torch.float32)
    other = hy.Hamiltonian(*synth.integrals(n, 714), n, na, nb)
    # T, 1,001 x 41 x 2,048 floats, and three states beside it
    ws = 1001 * 41 * 2048 * 4 + 3 * ham.n_det * 4
    filler = _leave(ws + 45 * MB)
    before = _free()
    other.apply_h(x, out=out)
    used = before - _free()
    del filler
    tol = 2e-5 * ref.abs().max().item()
    assert (out.double() - ref).abs().max().item() <= tol
    assert ws - 2 * MB <= used <= ws + 12 * MB
    assert torch.equal(other.apply_h(x), out)
