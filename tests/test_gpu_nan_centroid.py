"""A centroid with a NaN is never chosen, and the other lists are chosen as if
it were not there: the fused assignment, the one of few rows and an add with a
search of the nearest lists after it."""
import pytest

pytestmark = pytest.mark.gpu


def _index(torch, L, d, close, whole, dtypes=(), n_max=4096):
    from paper_2601_11808_gb300.sivf import Index
    g = torch.Generator(device="cuda")
    g.manual_seed(17)
    c = torch.randn((L, d), generator=g, device="cuda")
    if close:       # clusters of close centroids: the split first stage
        c = torch.randn((max(2, L // 16), d), generator=g, device="cuda")[torch.arange(L, device="cuda") % max(2, L // 16)] + 0.05 * c
    bad = L // 3
    if whole:
        c[bad] = float("nan")
    else:
        c[bad, d // 2] = float("nan")
    ix = Index(d, L, 32, n_max, n_max // 32 + 2 * L, scan_dtypes=dtypes)
    ix.set_centroids(c)
    return ix, c, bad, g


def _nearest(torch, x, c, bad):
    D = torch.cdist(x.double(), torch.nan_to_num(c).double(), compute_mode="donot_use_mm_for_euclid_dist")
    D[:, bad] = float("inf")
    return D.argmin(1).int()


@pytest.mark.parametrize("L,d,m,close", [
    (1024, 128, 12_000, False),    # fused, one product
    (1024, 128, 12_000, True),     # fused, split
    (1024, 128, 300, True),        # few rows
    (64, 32, 300, False),
    (300, 20, 200, False),         # the FP32 product
])
@pytest.mark.parametrize("whole", [False, True])
def test_assign(L, d, m, close, whole):
    import torch
    ix, c, bad, g = _index(torch, L, d, close, whole)
    x = torch.nan_to_num(c)[torch.arange(m, device="cuda") % L] + 0.3 * torch.randn((m, d), generator=g, device="cuda")
    got = ix.assign(x)
    ix.sync()
    assert torch.equal(got.int(), _nearest(torch, x, c, bad))
    ix.close()


@pytest.mark.parametrize("dtype", ["fp32", "bf16"])
def test_add_and_search(dtype):
    import torch
    L, d, n, k = 256, 64, 4096, 5
    ix, c, bad, g = _index(torch, L, d, False, True, ("bf16",))
    x = torch.nan_to_num(c)[torch.arange(n, device="cuda") % L] + 0.3 * torch.randn((n, d), generator=g, device="cuda")
    assert ix.add(torch.arange(n, device="cuda"), x, sync=True) == n
    assert int(ix.list_sizes()[bad]) == 0
    q = x[:100].contiguous()
    dist, lab = ix.search(q, k, 1, dtype=dtype)
    ix.sync()
    home = _nearest(torch, x, c, bad)
    D = torch.cdist(q.double(), x.double(), compute_mode="donot_use_mm_for_euclid_dist")
    D[home[:100, None] != home[None, :]] = float("inf")
    assert torch.equal(lab, D.topk(k, dim=1, largest=False).indices)
    ix.close()
