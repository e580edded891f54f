"""Grouping, seeding and numbering at the sizes where they change form: one CTA
up to 2,048 vertices, tiles of 2,048 sorted positions above, the queue order by
one block up to 4,096 clusters.  The refinement's result must be the oracle's."""
import numpy as np
import pytest

import oracle
import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _labels(kind, n, rng):
    if kind == "none":
        return np.full(n, -1, np.int32)
    if kind == "one":
        return np.full(n, 2**31 - 1, np.int32)
    if kind == "distinct":
        return rng.permutation(n).astype(np.int32)
    if kind == "pairs":  # n // 2 clusters: around the one-block order's limit
        return (rng.permutation(n) // 2).astype(np.int32)
    lab = rng.integers(0, max(1, n // 40), n).astype(np.int32)  # "mixed": some unclustered
    lab[rng.random(n) < 0.2] = -1
    return lab


@pytest.mark.parametrize("n", [1, 2, 33, 1023, 1024, 1025, 8191, 8192, 8193, 10_239, 10_240, 10_241])
@pytest.mark.parametrize("kind", ["none", "one", "distinct", "pairs", "mixed"])
def test_sizes(n, kind):
    import paper_2509_02590_gb300 as wcc
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    rng = np.random.default_rng(n)
    lab = _labels(kind, n, rng)
    m = min(3 * n, 6000 if kind == "one" else 3 * n)
    u, v = rng.integers(0, n, m), rng.integers(0, n, m)
    same = np.nonzero(lab >= 0)[0]
    if kind in ("pairs", "mixed") and len(same):  # edges inside the clusters
        order = same[np.argsort(lab[same], kind="stable")]
        u, v = np.concatenate([u, order[:-1]]), np.concatenate([v, order[1:]])
    src, dst = synth.graphs._dedup(n, u, v)
    off, adj = oracle.build_csr(n, src, dst)
    ref, _ = oracle.wcc(n, off, adj, lab, 2)
    with wcc.WccGraph.from_edges(src, dst, n) as g:
        dev = g.run(torch.from_numpy(lab).cuda(), min_size=2).cpu().numpy()
        host, st = g.run(lab, min_size=2, stats=True)
    assert np.array_equal(dev, ref) and np.array_equal(host, ref)
    assert st["in_clusters"] == len(np.unique(lab[lab >= 0]))


@pytest.mark.parametrize("n", [100, 9000])
def test_labels_below_minus_one_are_refused(n):
    import paper_2509_02590_gb300 as wcc
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    lab = np.zeros(n, np.int32)
    lab[n // 2] = -2
    with wcc.WccGraph.from_edges(np.array([0], np.int32), np.array([1], np.int32), n) as g:
        with pytest.raises(wcc.WccError):
            g.run(lab)


@pytest.mark.parametrize("n", [1000, 9000])
def test_device_output_that_only_a_copy_can_write(n):
    """clustering_out on the device path is written by the numbering kernel when
    it can; an address that is not aligned, or pinned host memory, takes a copy."""
    import paper_2509_02590_gb300 as wcc
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    w = synth.lfr_like(n, seed=3)
    lab = torch.from_numpy(w.labels).cuda()
    stream = torch.cuda.current_stream().cuda_stream
    with wcc.WccGraph.from_edges(w.src, w.dst, w.n) as g:
        ref = g.run(lab).cpu().numpy()
        for shift in (1, 2, 3):
            raw = torch.full((4 * n + 8,), 7, dtype=torch.uint8, device="cuda")
            torch.cuda.synchronize()
            wcc.wcc_run(g.handle, lab.data_ptr(), wcc.rule_struct(), 2, wcc.WCC_MODE_BATCHED,
                        raw.data_ptr() + shift, 1, stream, None)
            got = raw.cpu().numpy()
            assert np.array_equal(got[shift:shift + 4 * n].copy().view(np.int32), ref)
            assert (got[:shift] == 7).all() and (got[shift + 4 * n:] == 7).all()
        pinned = torch.empty(n, dtype=torch.int32).pin_memory()
        wcc.wcc_run(g.handle, lab.data_ptr(), wcc.rule_struct(), 2, wcc.WCC_MODE_BATCHED,
                    pinned.data_ptr(), 1, stream, None)
        assert np.array_equal(pinned.numpy(), ref)


@pytest.mark.parametrize("n", [2047, 2048, 2049, 4095, 4096, 4097])
@pytest.mark.parametrize("kind", ["none", "one", "distinct", "pairs", "mixed"])
def test_sizes_around_the_one_cta_limit(n, kind):
    test_sizes(n, kind)


@pytest.mark.parametrize("tiles", [32, 33, 34, 64, 65, 66, 500])
@pytest.mark.parametrize("over", [-1, 0, 1])
def test_running_counts_over_many_tiles(tiles, over):
    """The single-pass counts look back over 32 tiles of 2,048 positions at a
    time: numbering (representatives before a vertex) and grouping (clusters
    before a sorted position) at and around those sizes, with tiles that count
    nothing among them."""
    import paper_2509_02590_gb300 as wcc
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    n = 2048 * tiles + over
    rng = np.random.default_rng(n)
    v = np.arange(n)
    width = np.where(rng.random(n) < 0.5, 1, 5000)  # runs of one vertex, and longer than two tiles
    minima = np.zeros(n, np.int64)
    at = 0
    for w in width:
        if at >= n:
            break
        minima[at:at + w] = at
        at += w
    ref = np.cumsum(minima == v) - 1
    ids, k = torch.empty(n, dtype=torch.int32, device="cuda"), None
    mn = torch.from_numpy(minima.astype(np.int32)).cuda()
    k = wcc._binding.wcc_number_by_minima(mn.data_ptr(), n, ids.data_ptr(), 1,
                                          torch.cuda.current_stream().cuda_stream)
    want = ref[minima]
    assert k == int(ref[-1]) + 1 and np.array_equal(ids.cpu().numpy(), want)
    # the same runs as input clusters, joined up as paths: components in, components out
    same = np.nonzero(minima[1:] == minima[:-1])[0]
    perm = rng.permutation(n)
    src, dst = perm[same].astype(np.int32), perm[same + 1].astype(np.int32)
    lab = np.empty(n, np.int32)
    lab[perm] = minima
    with wcc.WccGraph.from_edges(torch.from_numpy(src).cuda(), torch.from_numpy(dst).cuda(), n) as g:
        out, st = g.run(torch.from_numpy(lab).cuda(), rule="linear", num=0, den=1, stats=True)
    assert st["in_clusters"] == k
    sizes = np.bincount(want)
    low = np.full(k, n)
    np.minimum.at(low, want, perm)
    order = np.argsort(low[sizes > 1])
    rank = np.full(k, -1)
    rank[np.nonzero(sizes > 1)[0][order]] = np.arange(len(order))
    got = out.cpu().numpy()
    assert np.array_equal(got[perm], rank[want])
