"""Two host threads, each with its own handles and stream, in the same kernels at
different sizes: a launch must not depend on the shared-memory size that the other
thread's launch of the same kernel asks for.  Every call succeeds and gives the bits
of the same call alone.
"""
import threading

import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _hpsi(dtype):
    def make(hy, cfg):
        n, na, nb = cfg
        ham = hy.Hamiltonian(*synth.integrals(n, 40 + n), n, na, nb)
        psi = torch.from_numpy(synth.random_state(ham.n_det, 1)).to("cuda", dtype)
        return lambda: ham.apply_h(psi)
    return make


def _screen(dtype):
    def make(hy, cfg):
        n, na, nb = cfg
        ham = hy.Hamiltonian(*synth.integrals(n, 40 + n), n, na, nb)
        pool = hy.Pool(ham)
        psi, sigma = (torch.from_numpy(synth.random_state(ham.n_det, s)).to("cuda", dtype) for s in (1, 2))
        return lambda: pool.gradients(psi, sigma)
    return make


def _evaluate(hy, cfg):
    n, length = cfg
    ham = hy.Hamiltonian(*synth.integrals(n, 40 + n), n, n // 2, n // 2)
    pool = hy.Pool(ham)
    rng = np.random.default_rng(1)
    ops, th = rng.integers(0, len(pool), length), 0.2 * rng.standard_normal(length)
    ad = hy.Adapt(ham, pool, "f64", max_iter=length)
    ad.set_ansatz(ops, th)

    def run():
        e, g = ad.evaluate(th, torch.float64)
        return torch.from_numpy(np.concatenate([[e], g]))
    return run


def _predict(hy, hidden):
    r = hy.Ranker(hidden=hidden, seed=3)
    x = torch.from_numpy(np.random.default_rng(2).standard_normal((65, 16)).astype(np.float32)).cuda()
    return lambda: r.predict(x)


# sizes beyond 48 KB of dynamic shared memory, and calls of each thread
CASES = {"hpsi_f64": (_hpsi(torch.float64), 4000, (12, 2, 6), (13, 1, 6)),
         "hpsi_f32": (_hpsi(torch.float32), 3000, (11, 2, 2), (11, 3, 5)),
         "screen_f64": (_screen(torch.float64), 4000, (12, 2, 6), (13, 2, 6)),
         "screen_f32": (_screen(torch.float32), 4000, (13, 2, 6), (14, 1, 7)),
         "evaluate": (_evaluate, 1500, (8, 60), (8, 90)),
         "predict": (_predict, 8000, 192, 256)}


@pytest.mark.parametrize("case", list(CASES))
def test_sizes_side_by_side(case):
    import __graft_entry__
    __graft_entry__.build()
    import paper_2604_01176_gb300 as hy
    make, calls, *cfgs = CASES[case]
    runs = [make(hy, c) for c in cfgs]
    ref = [r().clone() for r in runs]
    torch.cuda.synchronize()
    wrong = []

    def work(i):
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                for _ in range(calls):
                    out = runs[i]()
                torch.cuda.current_stream().synchronize()
                if not torch.equal(out, ref[i]):
                    wrong.append(f"{cfgs[i]}: other values")
        except Exception as e:              # noqa: BLE001 (reported below)
            wrong.append(f"{cfgs[i]}: {e}")

    threads = [threading.Thread(target=work, args=(i,)) for i in range(2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not wrong, wrong
