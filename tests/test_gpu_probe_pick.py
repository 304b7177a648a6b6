"""Probe selection from the split distances and their group minima at the
edges of its rule (L >= 32 P, P <= 128), of its tiles and segments, with exact
ties and with rows that have more candidates than a warp's table: the
oracle's FP64 set, listed nearest first."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind", ["apart", "close", "ties", "same"])
@pytest.mark.parametrize("d,L,P,m", [(16, 64, 2, 1), (32, 65, 2, 129), (64, 127, 3, 300), (96, 257, 8, 128),
                                     (128, 1000, 31, 200), (112, 1025, 32, 70), (128, 4096, 128, 33),
                                     (128, 4097, 100, 140), (64, 16400, 32, 5)])
def test_probe_sets_equal_the_oracle(d, L, P, m, kind):
    import torch
    from paper_2601_11808_gb300.sivf import Index
    rng = np.random.default_rng([d, L, P, m])
    if kind == "apart":
        c = 4.0 * rng.standard_normal((L, d))
        q = c[rng.integers(0, L, m)] + 0.5 * rng.standard_normal((m, d))
    elif kind == "close":
        base = rng.uniform(-1.0, 1.0, (3, d))
        c = base[rng.integers(0, 3, L)] + 0.05 * rng.standard_normal((L, d))
        q = base[rng.integers(0, 3, m)] + 0.05 * rng.standard_normal((m, d))
    elif kind == "ties":
        c, q = rng.integers(-1, 2, (L, d)), rng.integers(-1, 2, (m, d))
    else:
        c = np.repeat(rng.standard_normal((1, d)), L, 0)
        c[::7] += 1.0
        q = c[:1] + 0.01 * rng.standard_normal((m, d))
    c, q = c.astype(np.float32), q.astype(np.float32)
    g = Index(d, L, 32, 100, 10, 10)
    g.set_centroids(torch.from_numpy(c).cuda())
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


@pytest.mark.parametrize("d,L,P,m", [(128, 1000, 8, 2500), (96, 132, 4, 10001), (64, 100, 3, 40000),
                                     (32, 2049, 16, 1290)])
def test_probe_sets_where_a_range_of_steps_crosses_tiles(d, L, P, m):
    """More (tile, chunk) steps than the chip has SMs: ranges that begin and
    end inside a tile, take in a whole one, and rows of 16- and 32-byte
    alignment."""
    import torch
    from paper_2601_11808_gb300.sivf import Index
    rng = np.random.default_rng([d, L, P, m])
    c = rng.uniform(-1.0, 1.0, (L, d)).astype(np.float32)
    q = (c[rng.integers(0, L, m)] + 0.3 * rng.standard_normal((m, d))).astype(np.float32)
    g = Index(d, L, 32, 100, 10, 10)
    g.set_centroids(torch.from_numpy(c).cuda())
    o = oracle.OracleIVF(d, L, n_max=10, n_slabs=10)
    o.set_centroids(c)
    got = g.probe(torch.from_numpy(q).cuda(), P).cpu().numpy()
    g.sync()
    np.testing.assert_array_equal(np.sort(got, 1), np.sort(o.probe(q, P), 1))
    g.close()
