"""Pair pruning, the one-block grouping and the gathering merges against the
paths without them.

A query's farther lists whose vectors cannot lie within the bound its nearest
list left take no part in the scan.  Searches with pruning must return, bit
for bit, what the same search returns without it: reduced forms against the
single-launch tile (nearest_first = 0), the FP32 form against query batches
small enough for a single launch; both against the oracle's distances."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


def _cloud(rng, n, d, comps, spread):
    c = rng.uniform(-1.0, 1.0, (comps, d))
    x = c[rng.integers(0, comps, n)] + spread * rng.standard_normal((n, d))
    return c.astype(np.float32), x.astype(np.float32)


def _index(torch, d, L, C, cent, x, kinds=()):
    from paper_2601_11808_gb300.sivf import Index
    n = len(x)
    g = Index(d, L, C, 2 * n, 2 * (n // C + 2 * L), 0, kinds)
    g.set_centroids(torch.from_numpy(cent).cuda())
    g.add(torch.arange(n, device="cuda"), torch.from_numpy(x).cuda())
    return g


def _same(a, b):
    np.testing.assert_array_equal(a[1].cpu().numpy(), b[1].cpu().numpy())
    np.testing.assert_array_equal(a[0].cpu().numpy(), b[0].cpu().numpy())


# spread 0.02: separate clusters, most pairs pruned; 0.3: overlapping cells
@pytest.mark.parametrize("spread", [0.02, 0.3])
@pytest.mark.parametrize("d,L,C,P,k", [(32, 40, 32, 2, 1), (96, 65, 32, 17, 10), (128, 33, 64, 33, 7),
                                       (64, 24, 128, 5, 30)])
def test_reduced_forms_equal_the_unpruned_scan(d, L, C, P, k, spread):
    import torch
    rng = np.random.default_rng([d, L, P, int(100 * spread)])
    cent, x = _cloud(rng, 6000, d, L, spread)
    x[:50] *= 30.0                        # far members: their lists have a large radius
    q = torch.from_numpy(np.concatenate([x[rng.integers(0, 6000, 290)] + 0.01, 5.0 * cent[:10]])).cuda()
    g = _index(torch, d, L, C, cent, x, ("bf16", "fp8"))
    for form in ("bf16", "fp8"):
        for nq in (300, 1):
            got = g.search(q[:nq], k, P, form)
            cand = g.search_candidates(q[:nq], min(4 * k, 128), P, form)
            for shape in ((nq, k), (nq, max(1, min(4 * k, 128) // 4))):
                g.set_tile(form, shape[0], shape[1], P, {
                    "queries_per_tile": 64, "slabs_per_chunk": 4, "items_per_sm": 4,
                    "select_slabs": 0, "nearest_first": 0})
            _same(got, g.search(q[:nq], k, P, form))
            _same(cand, g.search_candidates(q[:nq], min(4 * k, 128), P, form))
            for shape in ((nq, k), (nq, max(1, min(4 * k, 128) // 4))):
                g.set_tile(form, shape[0], shape[1], P, None)
    g.close()


@pytest.mark.parametrize("spread", [0.02, 0.3])
@pytest.mark.parametrize("d,L,C,P,k", [(20, 40, 32, 8, 10), (100, 50, 64, 16, 24), (132, 30, 32, 9, 25),
                                       (256, 20, 32, 11, 72), (128, 64, 128, 64, 73),
                                       (4, 16, 32, 16, 300)])
def test_fp32_equals_the_single_launch_and_the_oracle(d, L, C, P, k, spread):
    import torch
    rng = np.random.default_rng([d, L, P, int(100 * spread), 1])
    cent, x = _cloud(rng, 5000, d, L, spread)
    nq = -(-2048 // P) + 3                # two launches; in parts of nq // 4, one
    qn = np.concatenate([x[rng.integers(0, 5000, nq - 2)] + np.float32(0.01), 4.0 * cent[:2]])
    q = torch.from_numpy(qn).cuda()
    g = _index(torch, d, L, C, cent, x)
    before = g.stats()["pairs_scanned"]
    got = g.search(q, k, P)
    scanned = g.stats()["pairs_scanned"] - before
    parts = [g.search(q[i:i + max(1, nq // 4)], k, P) for i in range(0, nq, max(1, nq // 4))]
    _same(got, [torch.cat([p[j] for p in parts]) for j in (0, 1)])
    once = g.stats()["pairs_scanned"] - before - scanned
    if spread < 0.1 and d >= 100:
        assert scanned < once             # clusters apart: pairs were pruned
    o = oracle.OracleIVF(d, L, C, 10_000, 2 * (5000 // C + 2 * L))
    o.set_centroids(cent)
    o.add(np.arange(5000), x)
    od, _ = o.search(qn[:40], k, P)
    gd = got[0][:40].cpu().numpy().astype(np.float64)
    fin = np.isfinite(od)
    assert (np.isfinite(gd) == fin).all()
    # (d + 1) u relative: the direct form's rounding
    assert (np.abs(gd - od)[fin] <= (d + 2) * 2.0 ** -24 * od[fin] + 1e-30).all()
    g.close()


def test_radii_follow_deletes_reloads_and_probe_lists(tmp_path):
    """A list emptied and refilled farther out, a loaded index, caller-given
    probes with repeats and gaps: the same results as a fresh index's."""
    import torch
    from paper_2601_11808_gb300.sivf import Index
    rng = np.random.default_rng(7)
    cent, x = _cloud(rng, 4000, 64, 30, 0.05)
    y = (x + 0.4 * rng.standard_normal(x.shape)).astype(np.float32)
    q = torch.from_numpy(np.concatenate([x[:200], y[:200]])).cuda()
    g = _index(torch, 64, 30, 32, cent, x, ("bf16", "fp8"))
    ids = torch.arange(4000, device="cuda")
    g.remove(ids, sync=True)
    g.add(ids, torch.from_numpy(y).cuda())
    fresh = _index(torch, 64, 30, 32, cent, y, ("bf16", "fp8"))
    g.save(str(tmp_path / "ix"))
    again = Index.load(str(tmp_path / "ix"))
    probes = torch.from_numpy(rng.integers(-1, 31, (400, 9)).astype(np.int32)).cuda()
    for form in ("fp32", "bf16", "fp8"):
        want = fresh.search(q, 10, 8, form)
        wantp = fresh.search_with_probes(q, 10, probes, form)
        for ix in (g, again):
            _same(ix.search(q, 10, 8, form), want)
            _same(ix.search_with_probes(q, 10, probes, form), wantp)
    for ix in (g, again, fresh):
        ix.close()


@pytest.mark.parametrize("k", [1, 10, 24, 25, 72, 73, 128])
def test_merges_of_many_equal_distances(k):
    """4,000 copies of one vector in one list cut into many chunks: more
    entries at the bound than a merge gathers; ties go to the lower id."""
    import torch
    cent = np.zeros((2, 32), np.float32)
    cent[1] = 1.0
    x = np.full((4000, 32), 0.25, np.float32)
    x[3000:] += np.float32(0.125)
    g = _index(torch, 32, 2, 32, cent, x, ("bf16", "fp8"))
    for nq in (1, 70):
        q = torch.zeros((nq, 32), device="cuda")
        for form in ("fp32", "bf16", "fp8"):
            dist, lab = g.search(q, k, 2, form)
            np.testing.assert_array_equal(dist.cpu().numpy(), np.full((nq, k), 2.0, np.float32))
            lab = lab.cpu().numpy()
            if form == "fp32":
                np.testing.assert_array_equal(lab, np.tile(np.arange(k), (nq, 1)))
            else:  # any 4k of the equal candidates: distinct, in order, among the near ones
                assert (np.diff(lab, axis=1) > 0).all() and lab.max() < 3000
    g.close()


@pytest.mark.parametrize("nq,P", [(1, 1), (1, 64), (1024, 8), (1025, 8), (8192, 1), (8193, 1), (127, 64),
                                  (129, 64), (1024, 2), (683, 3), (2048, 1), (2049, 1), (32, 64), (33, 64)])
def test_grouping_in_one_block_and_in_three(nq, P):
    """2,048 pairs group in one block, more in three launches."""
    import torch
    rng = np.random.default_rng([nq, P])
    cent, x = _cloud(rng, 3000, 16, 70, 0.3)
    qn = x[rng.integers(0, 3000, nq)] + np.float32(0.01)
    g = _index(torch, 16, 70, 32, cent, x, ("bf16",))
    o = oracle.OracleIVF(16, 70, 32, 6000, 1000)
    o.set_centroids(cent)
    o.add(np.arange(3000), x)
    m = min(nq, 200)
    od, _ = o.search(qn[-m:], 5, P)
    for form in ("fp32", "bf16"):
        gd, _ = g.search(torch.from_numpy(qn).cuda(), 5, P, form)
        gd = gd[-m:].cpu().numpy().astype(np.float64)
        # bf16: of 20 candidates the best 5 by exact distance; ranks by the
        # rounded form may miss one, so its distances are compared as a bound
        if form == "fp32":
            assert (np.abs(gd - od) <= 18 * 2.0 ** -24 * od + 1e-30).all()
        else:
            assert (gd >= od * (1 - 18 * 2.0 ** -24)).all()
            assert (np.abs(gd - od) <= 18 * 2.0 ** -24 * od + 1e-30).mean() > 0.95
    g.close()
