"""The ranker's forward pass at widths and row counts around its tile edges
(8 rows, 32 inputs, 256 units, 512 the widest single-launch width) against the
same network in 64 bits, and touched weights of one vector and of two in the
same launches against brute force.

Tolerance: a score sums at most 600 float products per layer over four layers
(the rounding of 600 terms, 600 x 2^-24 = 4e-5 of their absolute sum, typically
a twentieth of it): 1e-4 of the largest score.
"""
import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("hidden", [16, 40, 255, 256, 300, 512, 600])
@pytest.mark.parametrize("rows", [1, 7, 8, 65, 1107])
def test_forward_shapes(hidden, rows):
    import __graft_entry__
    __graft_entry__.build()
    import paper_2604_01176_gb300 as hy
    r = hy.Ranker(hidden=hidden, seed=3)
    w = r.params().astype(np.float64)
    x = np.random.default_rng(rows).standard_normal((rows, 16)).astype(np.float32)
    got = r.predict(torch.from_numpy(x).cuda()).cpu().numpy()
    z, fin, o = x.astype(np.float64), 16, 0
    for out in (hidden, hidden, hidden, 1):
        W = w[o:o + out * fin].reshape(out, fin)
        o += out * fin
        b = w[o:o + out]
        o += out
        z = z @ W.T + b
        if out != 1:
            z = np.maximum(z, 0.0)
        fin = out
    assert o == len(w)
    assert np.abs(got - z[:, 0]).max() <= 1e-4 * max(np.abs(z).max(), 1e-3)


@pytest.mark.parametrize("cfg", [(3, 1, 2), (6, 3, 3), (9, 5, 4), (12, 6, 6)])
def test_two_vectors_share_launches(cfg):
    """Features of (psi, sigma) use both vectors' weights from shared launches:
    the same as the features of psi with sigma's weights from its own call."""
    import __graft_entry__
    __graft_entry__.build()
    import paper_2604_01176_gb300 as hy
    n, na, nb = cfg
    ham = hy.Hamiltonian(*synth.integrals(n, 5), n, na, nb)
    pool = hy.Pool(ham)
    psi = torch.from_numpy(synth.random_state(ham.n_det, 1)).cuda()
    sigma = torch.from_numpy(synth.random_state(ham.n_det, 2)).cuda()
    both = hy.ranker_features(ham, pool, psi, sigma=sigma)
    again = hy.ranker_features(ham, pool, psi, sigma=sigma)
    assert torch.equal(both, again)
    swapped = hy.ranker_features(ham, pool, sigma, sigma=psi)
    alone = hy.ranker_features(ham, pool, psi)
    assert torch.isfinite(both).all() and torch.isfinite(swapped).all() and torch.isfinite(alone).all()
    d1, d2 = hy.touched_weights(ham, psi), hy.touched_weights(ham, sigma)
    w1, w2 = d1[0, 0].item(), d2[0, 0].item()
    assert abs(w1 - 1.0) <= 1e-5 and abs(w2 - 1.0) <= 1e-5


@pytest.mark.parametrize("hidden", [257, 384, 512])
@pytest.mark.parametrize("rows", [1, 255, 256, 257, 300])
def test_wide_network_few_rows(hidden, rows):
    """Beyond 256 units, up to 256 rows go through the products and more through the one
    launch: a row's score is the same bits in either (the first rows of 300 and of 257
    against the same rows alone)."""
    import __graft_entry__
    __graft_entry__.build()
    import paper_2604_01176_gb300 as hy
    r = hy.Ranker(hidden=hidden, seed=3)
    x = torch.from_numpy(np.random.default_rng(5).standard_normal((300, 16)).astype(np.float32)).cuda()
    assert torch.equal(r.predict(x[:rows].contiguous()), r.predict(x)[:rows])


def _touched(D, n, ann, cre):
    """Weight of one constituent's domain from D, as hyperion.h defines the feature:
    modes `ann` emptied and `cre` filled, in pairs."""
    a = [(x, y) for x, y in zip(ann, cre) if x < n]
    b = [(x - n, y - n) for x, y in zip(ann, cre) if x >= n]
    if len(a) <= 1 and len(b) <= 1:
        return max(D[a[0][0] * n + a[0][1] if a else 0, b[0][0] * n + b[0][1] if b else 0], 0.0)
    if not b:
        return np.sqrt(np.prod([max(D[x * n + y, 0], 0.0) for x, y in a]))
    return np.sqrt(np.prod([max(D[0, x * n + y], 0.0) for x, y in b]))


@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
@pytest.mark.parametrize("cfg", [(3, 1, 2), (6, 3, 3), (9, 5, 4), (12, 6, 6), (16, 3, 4), (16, 8, 2)],
                         ids=lambda c: "n%da%db%d" % c)
def test_second_vector_weights(cfg, dtype):
    """The two features that read both vectors' touched weights, from the shared
    launches, against 64-bit arithmetic on the weights of each vector from its own call
    (12,870 alpha strings: blocks of 16 rows and 160 threads).

    Tolerance: the bound and the weight sum at most four float terms of a few roundings
    each (1e-6 of them), log10 of values of up to 12 adds as much: 5e-6."""
    import __graft_entry__
    __graft_entry__.build()
    import paper_2604_01176_gb300 as hy
    n, na, nb = cfg
    ham = hy.Hamiltonian(*synth.integrals(n, 5), n, na, nb)
    pool = hy.Pool(ham)
    g = torch.Generator(device="cuda")
    g.manual_seed(n)
    v = torch.randn((2, ham.n_det), dtype=dtype, device="cuda", generator=g)
    v[1] *= torch.linspace(0.1, 2.0, ham.n_det, dtype=dtype, device="cuda")     # other weights
    psi, sigma = v[0].contiguous(), v[1].contiguous()
    feat = hy.ranker_features(ham, pool, psi, sigma=sigma).cpu().numpy().astype(np.float64)
    dp, ds = (hy.touched_weights(ham, x).cpu().numpy().astype(np.float64) for x in (psi, sigma))
    for k, d in enumerate(pool.descriptors()):
        bound = wsum = 0.0
        for c in range(d[0]):
            q = d[1 + 5 * c:6 + 5 * c]
            cre, ann = [q[1], q[2]][:q[0]], [q[4], q[3]][:q[0]]
            p, i = _touched(dp, n, ann, cre), _touched(dp, n, cre, ann)
            sp, si = _touched(ds, n, ann, cre), _touched(ds, n, cre, ann)
            bound += 2.0 * (np.sqrt(p * si) + np.sqrt(i * sp))
            wsum += p + i
        want = (np.log10(bound / np.sqrt(dp[0, 0] * ds[0, 0]) + 1e-12), np.log10(wsum / dp[0, 0] + 1e-12))
        assert np.abs(feat[k, 10:12] - want).max() <= 5e-6
