"""sivf_reserve for some number of probes covers every smaller one: the scratch
of a probe selection is not monotone in their number."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L,nq,k,reserved,probes", [
    (2048, 20_000, 1, 128, 64),     # 128 > L / 32
    (1024, 50_000, 10, 33, 32),
    (4096, 10_000, 10, 130, 128),   # 130 > 128
])
def test_fewer_probes_than_reserved(L, nq, k, reserved, probes):
    import torch
    from paper_2601_11808_gb300.sivf import Index
    g = torch.Generator(device="cuda")
    g.manual_seed(3)
    d, n = 128, 8 * L
    ix = Index(d, L, 32, n, 2 * (n // 32 + 2 * L))
    ix.set_centroids(torch.randn((L, d), generator=g, device="cuda"))
    ix.add(torch.arange(n, device="cuda"), torch.randn((n, d), generator=g, device="cuda"))
    q = torch.randn((nq, d), generator=g, device="cuda")
    warm, fresh = torch.cuda.Stream(), torch.cuda.Stream()
    torch.cuda.synchronize()
    with torch.cuda.stream(warm):          # modules and torch's own blocks
        want = ix.search(q, k, probes)
    torch.cuda.synchronize()
    with torch.cuda.stream(fresh):
        ix.reserve(max_queries=nq, max_k=k, max_nprobe=reserved)
        torch.cuda.synchronize()
        out = [torch.empty_like(t) for t in want]   # this stream's torch blocks
        del out
        torch.cuda.synchronize()
        free = torch.cuda.mem_get_info()[0]
        got = ix.search(q, k, probes)
        torch.cuda.synchronize()
        assert torch.cuda.mem_get_info()[0] == free
    for a, b in zip(want, got):
        assert torch.equal(a, b)
    ix.close()
