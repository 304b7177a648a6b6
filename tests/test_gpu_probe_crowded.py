"""Probe selection where hundreds of lists share a cluster: more of them lie
within the split products' bound of a row's P-th list than a warp's table
holds.  The oracle's FP64 set, nearest first, and a cost within a few times
that of lists that lie apart."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


def _crowded(rng, d, L, comps, m):
    """SIFT-like clusters with about L / comps trained centroids each."""
    base = rng.uniform(0.0, 255.0, (comps, d))
    c = base[np.arange(L) % comps] + 3.0 * rng.standard_normal((L, d))
    q = base[rng.integers(0, comps, m)] + 20.0 * rng.standard_normal((m, d))
    return c.astype(np.float32), q.astype(np.float32)


def _index(torch, c):
    from paper_2601_11808_gb300.sivf import Index
    g = Index(c.shape[1], len(c), 32, 100, 10, 10)
    g.set_centroids(torch.from_numpy(c).cuda())
    return g


# rows in one block and past it, one row a block and four, a last group cut short,
# a table for every list's number, one chunk of lists and several
@pytest.mark.parametrize("d,L,comps,P,m", [
    (16, 600, 1, 3, 5), (32, 2048, 2, 64, 61), (64, 705, 1, 16, 130), (96, 1000, 1, 2, 1),
    (112, 1999, 1, 8, 611), (128, 2048, 2, 32, 609), (128, 4097, 2, 100, 20), (128, 16390, 2, 7, 6)])
@pytest.mark.parametrize("ties", [False, True])
def test_crowded_probe_sets_equal_the_oracle(d, L, comps, P, m, ties):
    import torch
    rng = np.random.default_rng([d, L, P, m, ties])
    c, q = _crowded(rng, d, L, comps, m)
    if ties:  # a coarse grid: lists that are equal, distances that are equal
        c, q = 8.0 * np.rint(c / 8.0), np.rint(q)
        c[::3] = c[0]
    c, q = c.astype(np.float32), q.astype(np.float32)
    g = _index(torch, c)
    o = oracle.OracleIVF(d, L, n_max=10, n_slabs=10)
    o.set_centroids(c)
    got = g.probe(torch.from_numpy(q).cuda(), P).cpu().numpy()
    g.sync()
    np.testing.assert_array_equal(np.sort(got, 1), np.sort(o.probe(q, P), 1))
    far = ((q.astype(np.float64)[:, None] - c[got].astype(np.float64)) ** 2).sum(2)
    cn = (c.astype(np.float64) ** 2).sum(1)[got] + (q.astype(np.float64) ** 2).sum(1)[:, None]
    # nearest first up to the FP32 distances' error, 2 (d + 4) u (||q||^2 + ||c||^2) a pair
    assert (np.diff(far, axis=1) >= -4 * (d + 4) * 2.0 ** -24 * cn[:, 1:]).all()
    g.close()


def _us(torch, run):
    run()
    a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
    a.record()
    for _ in range(5):
        run()
    b.record()
    torch.cuda.synchronize()
    return a.elapsed_time(b) * 200.0


def test_crowded_probes_cost_a_few_times_the_others():
    """Deciding hundreds of lists per row by FP64 distance took 98 times as
    long as rows of lists that lie apart; in FP32 first, 6 times."""
    import torch
    rng = np.random.default_rng(1)
    us = []
    for comps in (2, 2048):
        c, q = _crowded(rng, 128, 2048, comps, 10_000)
        g, x = _index(torch, c), torch.from_numpy(q).cuda()
        us.append(_us(torch, lambda: g.probe(x, 32)))
        g.close()
    assert us[0] < 20.0 * us[1], us
