"""Float H|psi> with the same-spin parts on the tensor cores (512 and more
strings of each spin) against the FP32 pipes and the double sweep: ragged last
tiles of rows, columns and strings, one tile and many, ranges of rows that start
and end inside a tile; and its waits, which run out and are reported.

Tolerance: 2e-5 of the largest amplitude, the float sweep's bar in the parity
tests.
"""
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

# strings: 792 x 792, 924 x 792, 715 x 1287, 560 x 560, 1001 x 2002, 1820 x 560
CFGS = [(12, 5, 7), (12, 6, 5), (13, 9, 5), (16, 3, 13), (14, 4, 9), (16, 12, 3)]


def _ham(cfg):
    import __graft_entry__
    __graft_entry__.build()
    import paper_2604_01176_gb300 as hy
    n, na, nb = cfg
    ham = hy.Hamiltonian(*synth.integrals(n, 700 + n), n, na, nb)
    psi = torch.from_numpy(synth.random_state(ham.n_det, 9)).cuda().float()
    return hy, ham, psi


@pytest.mark.parametrize("cfg", CFGS, ids=["n%da%db%d" % c for c in CFGS])
def test_same_spin_matches_simt_and_double(cfg):
    hy, ham, psi = _ham(cfg)
    out = torch.full_like(psi, float("nan"))
    ham.apply_h(psi, out=out)
    ref = ham.apply_h(psi.double())
    ham.set_coupling("simt")
    simt = ham.apply_h(psi)
    ham.set_coupling("tensor")
    scale = ref.abs().max().item()
    assert (out - simt).abs().max().item() <= 2e-5 * scale
    assert (out.double() - ref).abs().max().item() <= 2e-5 * scale
    assert torch.equal(ham.apply_h(psi), out)
    na, nb = ham.n_alpha_str, ham.n_beta_str
    for a, b in ((0, 1), (1, 257), (255, 512), (300, na), (na - 1, na)):
        assert torch.equal(ham.apply_h_rows(psi, a, b), out[a * nb:b * nb])


def test_waits_run_out_and_are_reported():
    """One poll a wait: every role gives up at its first, what is in flight ends,
    the next call reports it and the handle then works."""
    hy, ham, psi = _ham((12, 5, 7))
    good = ham.apply_h(psi)
    ham.set_wait_limit(1)
    ham.apply_h(psi)
    torch.cuda.synchronize()
    ham.set_wait_limit(1 << 26)
    with pytest.raises(hy.HyError) as ei:
        ham.apply_h(psi)
    assert ei.value.status == 4 and "timed out" in str(ei.value)
    assert torch.equal(ham.apply_h(psi), good)


def test_captured_sweep_replays():
    """A sweep captured after a Hamiltonian's first float one (which makes the
    operands) replays to the same bits on new amplitudes."""
    hy, ham, psi = _ham((12, 6, 5))
    out = torch.empty_like(psi)
    ham.apply_h(psi, out=out)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        ham.apply_h(psi, out=out)
    new = torch.from_numpy(synth.random_state(ham.n_det, 10)).cuda().float()
    ref = ham.apply_h(new)
    psi.copy_(new)
    out.zero_()
    graph.replay()
    torch.cuda.synchronize()
    assert torch.equal(out, ref)


def test_first_tensor_sweep_captured():
    """The first sweep that asks for the tensor cores may be a captured one (the
    workspace is there from a sweep on the FP32 pipes): the graph runs the kernels that
    the calls beside it run, and gives their bits."""
    hy, ham, psi = _ham((12, 6, 5))
    out = torch.empty_like(psi)
    ham.set_coupling("simt")
    ham.apply_h(psi, out=out)
    ham.set_coupling("tensor")
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        ham.apply_h(psi, out=out)
    out.zero_()
    graph.replay()
    torch.cuda.synchronize()
    ref = ham.apply_h(psi)
    assert torch.equal(out, ref)
    nb = ham.n_beta_str
    assert torch.equal(ham.apply_h_rows(psi, 3, 300), out[3 * nb:300 * nb])
