"""Nearest-list assignment through the fused first stage (one launch over all
rows, no distance matrix) at the edges of its tiles: rows past a tile and
past one tile per SM, lists past a group of 16, a box of 128 and a chunk,
columns past the row.  The result is the oracle's FP64 assignment bit for
bit, whichever first stage the centroids select."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


def _inputs(kind, d, L, m):
    rng = np.random.default_rng([d, L, m])
    if kind == "apart":       # centroids far apart: the single product decides
        c = rng.standard_normal((L, d)) * 4.0
        x = c[rng.integers(0, L, m)] + 0.1 * rng.standard_normal((m, d))
    elif kind == "close":     # centroids close against their norms: the split
        base = rng.uniform(-1.0, 1.0, (4, d))
        c = base[rng.integers(0, 4, L)] + 0.1 * rng.standard_normal((L, d))
        x = base[rng.integers(0, 4, m)] + 0.1 * rng.standard_normal((m, d))
    elif kind == "ties":      # integer grid: exact ties, several candidates a row
        c = rng.integers(-2, 3, (L, d))
        x = rng.integers(-2, 3, (m, d))
    else:                     # "same": one point repeated, every list qualifies
        c = np.repeat(rng.standard_normal((1, d)), L, 0)
        c[L // 2] += 1.0
        x = c[:1] + 0.01 * rng.standard_normal((m, d))
    return c.astype(np.float32), x.astype(np.float32)


@pytest.mark.parametrize("kind,d,L,m", [
    ("apart", 16, 16, 1), ("close", 16, 17, 129), ("ties", 32, 33, 128), ("same", 32, 40, 300),
    ("apart", 64, 127, 152 * 128 + 1), ("close", 64, 129, 700), ("ties", 80, 256, 2000),
    ("apart", 112, 257, 127), ("close", 128, 1000, 2 * 152 * 128 + 77), ("close", 96, 2049, 1500),
    ("ties", 128, 511, 1000), ("same", 128, 300, 200), ("apart", 128, 4096, 300),
    ("close", 128, 4095, 513)])
def test_assignment_equals_the_oracle(kind, d, L, m):
    import torch
    from paper_2601_11808_gb300.sivf import Index
    cent, x = _inputs(kind, d, L, m)
    g = Index(d, L, 32, 100, 10, 10)
    g.set_centroids(torch.from_numpy(cent).cuda())
    o = oracle.OracleIVF(d, L, n_max=10, n_slabs=10)
    o.set_centroids(cent)
    got = g.assign(torch.from_numpy(x).cuda()).cpu().numpy()
    np.testing.assert_array_equal(got, o.assign(x))
    g.sync()  # no sticky device error
    g.close()
