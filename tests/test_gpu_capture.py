"""Calls captured after a first hy_apply_h of their precision, which makes the handle's
workspace: the graph's results are those of the calls by themselves.  Sizes: those whose
own sweep needs no workspace, and one beyond (3,003 beta strings)."""
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
@pytest.mark.parametrize("cfg", [(6, 3, 3), (10, 4, 5), (12, 5, 6), (15, 2, 5)], ids=lambda c: "n%da%db%d" % c)
def test_after_a_first_sweep(cfg, dtype):
    import __graft_entry__
    __graft_entry__.build()
    import paper_2604_01176_gb300 as hy
    n, na, nb = cfg
    ham = hy.Hamiltonian(*synth.integrals(n, 60 + n), n, na, nb)
    psi = torch.from_numpy(synth.random_state(ham.n_det, 1)).to("cuda", dtype)
    sigma = ham.apply_h(psi)
    out, e, d = torch.empty_like(psi), torch.zeros((), dtype=torch.float64, device="cuda"), \
        torch.zeros((), dtype=torch.float64, device="cuda")
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        ham.apply_h(psi, out=out)
        ham.energy(psi, out, out=e)
        ham.dot(psi, psi, out=d)
    graph.replay()
    torch.cuda.synchronize()
    assert torch.equal(out, sigma)
    assert e.item() == ham.energy(psi, sigma).item() and d.item() == ham.dot(psi, psi).item()


@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
def test_operator_list_after_a_whole_screen(dtype):
    import __graft_entry__
    __graft_entry__.build()
    import paper_2604_01176_gb300 as hy
    n, na, nb = 10, 5, 5
    ham = hy.Hamiltonian(*synth.integrals(n, 60 + n), n, na, nb)
    pool = hy.Pool(ham)
    psi, sigma = (torch.from_numpy(synth.random_state(ham.n_det, s)).to("cuda", dtype) for s in (1, 2))
    pool.gradients(psi, sigma)
    ops = torch.tensor([3, 0, len(pool) - 1], dtype=torch.int32, device="cuda")
    g = torch.zeros(3, dtype=torch.float64, device="cuda")
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        pool.gradients(psi, sigma, ops=ops, out=g)
    graph.replay()
    torch.cuda.synchronize()
    assert torch.equal(g, pool.gradients(psi, sigma, ops=ops))


@pytest.mark.parametrize("hidden", [40, 300, 512])
def test_few_rows_of_a_ranker_after_many(hidden):
    """A wide network's products have their buffers from the first call, whatever its
    rows; and a first call may be a captured one."""
    import __graft_entry__
    __graft_entry__.build()
    import paper_2604_01176_gb300 as hy
    x = torch.randn((600, 16), device="cuda")
    few = x[:9].contiguous()
    for warm in (True, False):
        r = hy.Ranker(hidden=hidden, seed=3)
        if warm:
            r.predict(x)
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            out = r.predict(few)
        graph.replay()
        torch.cuda.synchronize()
        assert torch.equal(out, r.predict(few))
