"""Calls with little device memory left: scratch that does not fit is done without, and
nothing is held that is not used.  The rest of the device is filled by one tensor.
"""
import contextlib

import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

MB = 1 << 20


def _free():
    torch.cuda.synchronize()
    return torch.cuda.mem_get_info()[0]


@contextlib.contextmanager
def _leave(nbytes):
    """The device filled up to about nbytes."""
    torch.cuda.empty_cache()
    filler = torch.empty(_free() - nbytes, dtype=torch.uint8, device="cuda")
    try:
        yield
    finally:
        del filler
        torch.cuda.empty_cache()


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
    with _leave(ws + 45 * MB):
        before = _free()
        other.apply_h(x, out=out)
        used = before - _free()
    tol = 2e-5 * ref.abs().max().item()
    assert (out.double() - ref).abs().max().item() <= tol
    assert ws - 2 * MB <= used <= ws + 12 * MB
    assert torch.equal(other.apply_h(x), out)


def test_support_rows_without_tables():
    """A double sparse evaluation beyond the support programs (16 orbitals, 1 + 8
    electrons: 140 MB of tables) with 100 MB left.  Tolerances: energies 1e-10,
    gradients 1e-9, as for the other sparse evaluations."""
    import __graft_entry__
    __graft_entry__.build()
    import paper_2604_01176_gb300 as hy
    n, na, nb = 16, 1, 8
    ham = hy.Hamiltonian(*synth.integrals(n, 900 + n), n, na, nb)
    pool = hy.Pool(ham)
    sp = hy.Adapt(ham, pool, "f64", max_iter=160, sparse=True, sparse_cap=ham.n_det)
    de = hy.Adapt(ham, pool, "f64", max_iter=160)
    rng = np.random.default_rng(17)
    for length in range(20, 161, 20):
        ops = [int(k) for k in rng.choice(len(pool), length)]
        th = rng.uniform(0.1, 0.7, length)
        de.set_ansatz(ops, th)
        ref = de.evaluate(th, torch.float64)
        if int((de.state(torch.float64) != 0).sum()) > 65536:
            break
    else:
        pytest.fail("no support beyond the programs")
    sp.set_ansatz(ops, th)
    with _leave(100 * MB):
        for _ in range(2):
            e, g = sp.evaluate(th, torch.float64)
            assert abs(e - ref[0]) < 1e-10
            assert np.abs(np.asarray(g) - np.asarray(ref[1])).max() < 1e-9


def test_ranker_buffers_half_allocated():
    """A fit whose batch does not fit leaves the ranker able to predict."""
    import __graft_entry__
    __graft_entry__.build()
    import paper_2604_01176_gb300 as hy
    r = hy.Ranker(hidden=600, seed=3)
    x = torch.from_numpy(np.random.default_rng(1).standard_normal((4096, 16)).astype(np.float32)).cuda()
    ref = r.predict(x)
    r.add_samples(x, x[:, 0].double().contiguous())
    with _leave(700 * MB):
        with pytest.raises(hy.HyError) as ei:
            r.fit(epochs=1, batch=1 << 17)
        assert ei.value.status == 3
        assert torch.equal(r.predict(x), ref)
    assert torch.equal(r.predict(x), ref)
