"""Nearest-list assignment where many lists share a cluster, as after training:
more lists than an undecided row's record holds lie within the products' bound
of its nearest, in either form of the first stage, at the edges of the second
pass's tiles and of the rule between the fused stage and the one for few rows.
The oracle's FP64 assignment bit for bit, and a cost within a few times that of
lists that lie apart."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


def _inputs(rng, form, d, L, comps, m):
    if form == "same":        # one point repeated: every list qualifies
        c = np.repeat(rng.standard_normal((1, d)), L, 0)
        c[L // 2] += 1.0
        x = c[:1] + 0.01 * rng.standard_normal((m, d))
        return c.astype(np.float32), x.astype(np.float32)
    base = rng.uniform(0.0, 255.0, (comps, d))
    c = base[np.arange(L) % comps] + 3.0 * rng.standard_normal((L, d))
    x = base[rng.integers(0, comps, m)] + 20.0 * rng.standard_normal((m, d))
    if form == "single":      # most lists far apart: the spacing chooses the single product
        far = rng.permutation(L)[:int(0.6 * L)]
        c[far] = rng.uniform(0.0, 255.0, (len(far), d))
    if form == "ties":
        c, x = 8.0 * np.rint(c / 8.0), np.rint(x)
    return c.astype(np.float32), x.astype(np.float32)


def _index(torch, c):
    from paper_2601_11808_gb300.sivf import Index
    g = Index(c.shape[1], len(c), 32, 100, 10, 10)
    g.set_centroids(torch.from_numpy(c).cuda())
    return g


@pytest.mark.parametrize("form,d,L,comps,m", [
    ("split", 128, 512, 4, 1), ("split", 128, 4096, 2, 129), ("split", 64, 257, 1, 5120),
    ("split", 64, 257, 1, 5121), ("split", 128, 600, 2, 152 * 128 + 1), ("split", 96, 4095, 16, 5300),
    ("single", 128, 400, 1, 2560), ("single", 128, 400, 1, 2561), ("single", 32, 1000, 2, 20000),
    ("single", 112, 129, 1, 6001), ("ties", 128, 300, 2, 5500), ("ties", 32, 900, 1, 300),
    ("same", 128, 300, 1, 5200), ("same", 48, 70, 1, 200)])
def test_crowded_assignment_equals_the_oracle(form, d, L, comps, m):
    import torch
    from paper_2601_11808_gb300 import sivf
    rng = np.random.default_rng([d, L, m, len(form)])
    c, x = _inputs(rng, form, d, L, comps, m)
    g = _index(torch, c)
    if form in ("single", "split"):
        assert sivf.sivf_assign_stage(g.h) == (1 if form == "single" else 3)
    o = oracle.OracleIVF(d, L, n_max=10, n_slabs=10)
    o.set_centroids(c)
    got = g.assign(torch.from_numpy(x).cuda()).cpu().numpy()
    np.testing.assert_array_equal(got, o.assign(x))
    g.sync()  # no sticky device error
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


@pytest.mark.parametrize("L,comps,m", [(512, 16, 200_000), (4096, 16, 10_000), (4096, 16, 300)])
def test_crowded_rows_cost_a_few_times_the_others(L, comps, m):
    """Rows recomputed from every list took 40 to 90 times as long as rows of
    lists that lie apart; by the second pass, 1 to 6 times."""
    import torch
    rng = np.random.default_rng(1)
    us = []
    for n in (comps, L):
        c, x = _inputs(rng, "split", 128, L, n, m)
        g, x = _index(torch, c), torch.from_numpy(x).cuda()
        us.append(_us(torch, lambda: g.assign(x)))
        g.close()
    assert us[0] < 12.0 * us[1], us
