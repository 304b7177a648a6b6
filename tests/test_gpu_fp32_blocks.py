"""The FP32 scan's selection by blocks: lists shorter and longer than a block,
swizzled (d % 32 == 0) and plain slabs, every tile, ties across a block's end
and holes left by deletes, against the oracle and against each other."""
import numpy as np
import pytest

import oracle
from sivf_check import compare_topk

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,C", [(32, 32), (64, 128), (128, 64), (96, 32), (20, 128), (100, 64), (160, 128),
                                 (256, 64)])
@pytest.mark.parametrize("k", [1, 10, 60, 200])
def test_blocks_tiles_and_ties(d, C, k):
    import torch
    from paper_2601_11808_gb300.sivf import Index
    rng = np.random.default_rng([d, C, k])
    L, n = 5, 4200                       # the first list: 3,400 rows, more than a block
    cent = (8.0 * rng.standard_normal((L, d))).astype(np.float32)
    lab = np.where(rng.random(n) < 0.8, 0, rng.integers(0, L, n))
    # small integers around the centroids: many equal distances
    x = (np.rint(cent[lab]) + rng.integers(-1, 2, (n, d))).astype(np.float32)
    S = 2 * (n // C + 2 * L)
    g = Index(d, L, C, 2 * n, S)
    o = oracle.OracleIVF(d, L, C, 2 * n, S)
    for ix, to in ((g, lambda a: torch.from_numpy(a).cuda()), (o, lambda a: a)):
        ix.set_centroids(to(cent))
        ix.add(to(np.arange(n, dtype=np.int64)), to(x))
        ix.remove(to(np.arange(0, n, 3, dtype=np.int64)))
    q = np.rint(cent[rng.integers(0, L, 70)]).astype(np.float32)
    od, oi = o.search(q, k, 3)
    want = None
    for tq in (0, 8, 16, 32, 64):
        if tq:
            tile = {"queries_per_tile": tq, "slabs_per_chunk": 16, "items_per_sm": 1,
                    "select_slabs": 0, "nearest_first": 0}
            try:
                g.set_tile("fp32", 70, k, 3, tile)
            except Exception:
                continue                 # over shared memory for this shape
        gd, gi = (t.cpu().numpy() for t in g.search(torch.from_numpy(q).cuda(), k, 3))
        fin = np.isfinite(od)
        assert (np.isfinite(gd) == fin).all()
        # integers: every FP32 sum of squares is exact
        np.testing.assert_array_equal(gd[fin].astype(np.float64), od[fin])
        np.testing.assert_array_equal(gi, oi)
        want = (gd, gi) if want is None else want
        np.testing.assert_array_equal(gd, want[0])
    g.close()


@pytest.mark.parametrize("C,d,tq,sl,k", [(32, 40, 64, 0, 192), (64, 96, 64, 2, 64), (64, 128, 64, 2, 10)])
def test_tiles_without_room_for_a_block_are_narrowed(C, d, tq, sl, k):
    """Tiles that fit 220 KB with the slabs' ids, but not beside a block's
    distances, are accepted and give the oracle's results; one above 220 KB is
    refused."""
    import torch
    from paper_2601_11808_gb300.sivf import Index
    rng = np.random.default_rng([C, d, tq, sl, k])
    L, n = 4, 3000
    cent = (8.0 * rng.standard_normal((L, d))).astype(np.float32)
    x = (np.rint(cent[rng.integers(0, L, n)]) + rng.integers(-1, 2, (n, d))).astype(np.float32)
    S = 2 * (n // C + 2 * L)
    g = Index(d, L, C, 2 * n, S)
    o = oracle.OracleIVF(d, L, C, 2 * n, S)
    for ix, to in ((g, lambda a: torch.from_numpy(a).cuda()), (o, lambda a: a)):
        ix.set_centroids(to(cent))
        ix.add(to(np.arange(n, dtype=np.int64)), to(x))
    q = np.rint(cent[rng.integers(0, L, 70)]).astype(np.float32)
    tile = {"queries_per_tile": tq, "slabs_per_chunk": 2, "items_per_sm": 4, "select_slabs": sl,
            "nearest_first": 0}
    g.set_tile("fp32", 70, k, 2, tile)
    assert g.get_tile("fp32", 70, k, 2)["queries_per_tile"] == tq
    gd, gi = (t.cpu().numpy() for t in g.search(torch.from_numpy(q).cuda(), k, 2))
    od, oi = o.search(q, k, 2)
    np.testing.assert_array_equal(gd.astype(np.float64), od)
    np.testing.assert_array_equal(gi, oi)
    with pytest.raises(Exception):
        g.set_tile("fp32", 70, 1000, 2, dict(tile, queries_per_tile=64, select_slabs=8))
    g.close()


def test_allocation_free_search_at_its_scratch_limit():
    """Eleven pairs per list: the 16-query tile's runs do not fit the fixed
    scratch, the 8-query tile's do."""
    import torch
    from paper_2601_11808_gb300 import sivf
    rng = np.random.default_rng(5)
    d, L, n, nq, k, P = 16, 2048, 6000, 186, 100, 128
    cent = (4.0 * rng.standard_normal((L, d))).astype(np.float32)
    x = (cent[rng.integers(0, L, n)] + rng.standard_normal((n, d))).astype(np.float32)
    g = sivf.Index(d, L, 32, 2 * n, 4096)
    g.set_centroids(torch.from_numpy(cent).cuda())
    g.add(torch.arange(n, device="cuda"), torch.from_numpy(x).cuda())
    q = torch.from_numpy(x[:nq]).cuda()
    want = g.search(q, k, P)
    dist = torch.empty((nq, k), dtype=torch.float32, device="cuda")
    lab = torch.empty((nq, k), dtype=torch.int64, device="cuda")
    sivf.sivf_search_noalloc(g.h, q, k, P, dist, lab)
    g.sync()
    compare_topk(dist.cpu().numpy(), lab.cpu().numpy(), want[0].cpu().numpy(), want[1].cpu().numpy())
    g.close()
