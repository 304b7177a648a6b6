"""The order of a row's probes: nearest first by FP32 distances whose sums are
fixed (in order over the coordinates; for at most 8 of at most 4,096 lists a
float4 per lane and a butterfly over the warp), ties to the lower list.  A form
of the selection that sums otherwise returns the same order."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _fma(a, b, c):  # exact products, one rounding (the FP64 one is 29 bits finer)
    return (a.astype(np.float64) * b.astype(np.float64) + c.astype(np.float64)).astype(np.float32)


def _distances(q, c, cn, warp):
    """fl(||c||^2 - 2 q.c) of rows q[m, 1, d] and their lists c[m, P, d]."""
    m, P, d = c.shape
    if warp:
        s = np.zeros((m, P, 32), np.float32)
        for j in range(d):
            s[..., j // 4] = _fma(q[..., j], c[..., j], s[..., j // 4])
        for o in (16, 8, 4, 2, 1):
            s = s + s[..., np.arange(32) ^ o]
        dot = s[..., 0]
    else:
        dot = np.zeros((m, P), np.float32)
        for j in range(d):
            dot = _fma(q[..., j], c[..., j], dot)
    return _fma(np.full((m, P), -2.0, np.float32), dot, cn)


@pytest.mark.parametrize("d,L,comps,P,m", [
    (128, 2048, 16, 32, 300), (96, 1024, 16, 16, 61), (128, 512, 16, 8, 700), (64, 4096, 128, 4, 130),
    (128, 4096, 128, 64, 200), (32, 8192, 256, 4, 40), (128, 1024, 8, 9, 40), (128, 200, 8, 8, 300),
    (112, 300, 8, 12, 50)])
def test_probes_are_ordered_by_fixed_sums(d, L, comps, P, m):
    import torch
    from paper_2601_11808_gb300.sivf import Index
    rng = np.random.default_rng([d, L, P, m])
    base = rng.uniform(0.0, 255.0, (comps, d))
    c = (base[np.arange(L) % comps] + 5.0 * rng.standard_normal((L, d))).astype(np.float32)
    q = (base[rng.integers(0, comps, m)] + 20.0 * rng.standard_normal((m, d))).astype(np.float32)
    g = Index(d, L, 32, 100, 10, 10)
    g.set_centroids(torch.from_numpy(c).cuda())
    got = g.probe(torch.from_numpy(q).cuda(), P).cpu().numpy()
    g.sync()
    lists = np.sort(got, 1)
    cn = (c.astype(np.float64) ** 2).sum(1).astype(np.float32)[lists]
    key = _distances(q[:, None], c[lists], cn, P <= 8 and L <= 4096)
    want = np.take_along_axis(lists, np.argsort(key, axis=1, kind="stable"), 1)
    np.testing.assert_array_equal(got, want)
    g.close()
