"""Pruned pairs at the ends of FP32's range: a large batch, whose farther lists
are pruned, finds what batches too small for that find."""
import pytest

pytestmark = pytest.mark.gpu


def _both(torch, ix, q, k, P):
    dist, lab = ix.search(q, k, P)
    few = 512 // P
    parts = [ix.search(q[i:i + few].contiguous(), k, P) for i in range(0, len(q), few)]
    ix.sync()
    return dist, lab, torch.cat([p[0] for p in parts]), torch.cat([p[1] for p in parts])


@pytest.mark.parametrize("c0,x0,x1,q,c1,best", [
    # ||q - c||^2 overflows for the list that holds the nearest vector
    ((5.7124527e18, 7.5753156e17, 8.7404955e17, -6.4225292e17),
     (8.6211078e17, 3.3002982e18, 4.8099181e18, 4.1460648e18),
     (-5.1375885e18, -3.2742747e18, -2.0074443e18, 4.9679212e18),
     (-2.522659e18, -5.210937e18, -6.153209e17, -9.918200e18),
     (-2.8946631e18, -3.9307486e17, -7.3986316e17, 8.2473405e18), 1),
    # the squares of the list's radius are rounded below the range
    ((-2.9542671768748813e-22, 1.0855195428079729e-23, 3.559996421085987e-23, 3.2939991502770657e-22),
     (-8.382583022551205e-23, -3.1289187093714062e-22, 1.4774439578719908e-22, 3.87095964701672e-22),
     (-2.06538457799698e-23, -4.270198348839511e-24, -6.625496014822907e-24, 2.117789081247355e-23),
     (-2.9932174680600946e-22, -6.188499574399762e-23, -9.601868525766147e-23, 3.0691636948694905e-22),
     (0.0, 0.0, 0.0, 0.0), 1),
    ((6.842662164509924e-23, 8.777602280941368e-23, 1.9448408887718194e-22, -1.856634122664606e-22),
     (2.7648110602156374e-22, 3.8886967742629436e-23, 3.061315980366607e-22, -1.4514564815168588e-22),
     (7.401161643682287e-24, 4.164703979984305e-24, 1.3005971832484168e-23, -1.8505357861051407e-23),
     (8.405742085462321e-23, 4.7299910550434615e-23, 1.477130937864799e-22, -2.1017141470373043e-22),
     (0.0, 0.0, 0.0, 0.0), 1),
])
def test_the_nearest_vector_of_the_farther_list(c0, x0, x1, q, c1, best):
    import torch
    from paper_2601_11808_gb300.sivf import Index
    ix = Index(4, 2, 32, 64, 16)
    ix.set_centroids(torch.tensor([c0, c1], device="cuda"))
    ix.add(torch.arange(2, device="cuda"), torch.tensor([x0, x1], device="cuda"))
    assert ix.list_sizes().tolist() == [1, 1]
    dist, lab, dist1, lab1 = _both(torch, ix, torch.tensor([q], device="cuda").repeat(1024, 1), 1, 2)
    assert (lab1 == best).all() and torch.equal(lab, lab1) and torch.equal(dist, dist1)
    ix.close()


@pytest.mark.parametrize("scale", [3e-22, 1e-19])
def test_squares_below_the_range(scale):
    import torch
    from paper_2601_11808_gb300.sivf import Index
    g = torch.Generator(device="cuda")
    g.manual_seed(7)
    d, L, n, nq, k, P = 4, 16, 4000, 2048, 3, 16
    r = lambda m: torch.randn((m, d), generator=g, device="cuda") * scale
    ix = Index(d, L, 32, n, 2 * (n // 32 + 2 * L))
    ix.set_centroids(4 * r(L))
    ix.add(torch.arange(n, device="cuda"), 4 * r(n))
    dist, _, dist1, _ = _both(torch, ix, 4 * r(nq), k, P)
    assert torch.equal(dist, dist1)
    ix.close()
