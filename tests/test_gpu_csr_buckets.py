"""The device CSR builder at the sizes where it changes form, against the
oracle's CSR: the one-CTA build and its limits, one and two partition digits,
rows around the register sort, the parts and the shared-memory limits, large
buckets, and rows that only the full sort takes (too many equal columns)."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _random(n, m, seed, lo=0):
    rng = np.random.default_rng(seed)
    return rng.integers(lo, n, m), rng.integers(lo, n, m)


def _hubs(n, m, rows, seed, span=None):
    """m random edges plus hubs of the given numbers of distinct neighbours
    (drawn from the first span vertices past the hubs)."""
    rng = np.random.default_rng(seed)
    u, v = _random(n, m, seed + 1, len(rows))
    us, vs = [u], [v]
    for h, d in enumerate(rows):
        hi = n if span is None else len(rows) + span
        us.append(np.full(d, h))
        vs.append(rng.choice(np.arange(len(rows), hi), size=d, replace=False))
    return np.concatenate(us), np.concatenate(vs)


CASES = {
    # one CTA: no edges left, its largest sizes, one more entry, one more row
    "loops": (5, np.arange(5), np.arange(5)),
    "two": (2, np.array([1, 0, 1]), np.array([0, 1, 1])),
    "small": (300, *_random(300, 2000, 1)),
    "small_full": (4096, *_random(4096, 6144, 2)),
    "small_over": (4096, *_random(4096, 6145, 3)),
    "small_rows_over": (4097, *_random(4097, 6000, 4)),
    "small_dense": (40, *_random(40, 6000, 5)),
    "small_hub": (4096, *_hubs(4096, 100, [511, 512, 513, 1500, 3000], 6)),
    # one digit: a single row per bucket, few rows, the most buckets
    "dense": (64, *_random(64, 200_000, 7)),
    "one_digit": (70_001, *_random(70_001, 400_000, 8)),
    "one_digit_last": (1023 * 256, *_random(1023 * 256, 300_000, 9)),
    # two digits from the next bucket on
    "two_digits": (1023 * 256 + 1, *_random(1023 * 256 + 1, 300_000, 10)),
    "two_digits_odd": (700_003, *_random(700_003, 900_001, 11)),
    # rows around the parts, the register sort and a CTA's shared memory
    "rows": (50_000, *_hubs(50_000, 60_000, [255, 256, 257, 383, 384, 385, 511, 512, 513, 767, 769,
                                             1025, 6143, 12_287], 12)),
    "large": (60_000, *_hubs(60_000, 60_000, [12_288, 12_289, 16_383, 16_384, 16_385, 59_000], 13)),
    # columns crowded into one part: sorted by the CTA
    "crowded": (60_000, *_hubs(60_000, 60_000, [3000, 12_000, 16_000], 14, span=16_100)),
    # more copies of one edge than a CTA sorts: the full sort
    "copies": (30_000, np.concatenate([np.full(40_000, 7), _random(30_000, 30_000, 15)[0]]),
               np.concatenate([np.full(40_000, 9), _random(30_000, 30_000, 15)[1]])),
}


@pytest.mark.parametrize("name", list(CASES))
@pytest.mark.parametrize("on_device", [True, False])
def test_builder_equals_oracle(name, on_device):
    import paper_2509_02590_gb300 as wcc
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    n, u, v = CASES[name]
    src, dst = u.astype(np.int32), v.astype(np.int32)
    off, adj = oracle.build_csr(n, src, dst)
    if on_device:
        src, dst = torch.from_numpy(src).cuda(), torch.from_numpy(dst).cuda()
    with wcc.WccGraph.from_edges(src, dst, n) as g:
        goff, gadj = g.csr()
    assert np.array_equal(goff, off) and np.array_equal(gadj, adj)


@pytest.mark.parametrize("n,m", [(100, 50), (100_000, 300_000), (400_000, 300_000)])
@pytest.mark.parametrize("bad", [-1, "n"])
def test_builder_refuses_endpoints_out_of_range(n, m, bad):
    import paper_2509_02590_gb300 as wcc
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    u, v = _random(n, m, 20)
    u[m // 2] = n if bad == "n" else bad
    with pytest.raises(wcc.WccError):
        wcc.WccGraph.from_edges(u.astype(np.int32), v.astype(np.int32), n)


HUGE = 32_768  # entries of a bucket that one CTA takes; more are sorted together
HUGE_CASES = {
    # rows (a bucket of their own entries and few more) around the limit
    "rows": (300_000, *_hubs(300_000, 400_000, [HUGE - 300, HUGE - 1, HUGE, HUGE + 1, 70_000], 31)),
    # one digit, two digits; one huge bucket, many, hubs in the last rows
    "one_digit": (100_000, *_hubs(100_000, 300_000, [99_000], 32)),
    "many": (400_000, *_hubs(400_000, 500_000, [60_000 + 1000 * k for k in range(12)], 33)),
    "last_rows": (300_000, *(299_999 - x for x in _hubs(300_000, 200_000, [200_000, 40_000], 34))),
    "star": (250_000, np.zeros(249_999, np.int64), np.arange(1, 250_000)),
    # equal columns past what a CTA sorts: below the limit, and above with loops and repeats
    "copies_below": (30_000, *(np.concatenate([np.full(17_000, a), b]) for a, b in
                               zip((7, 9), _random(30_000, 30_000, 35)))),
    "copies_above": (30_000, *(np.concatenate([np.full(90_000, a), np.full(300, 5), b]) for a, b in
                               zip((7, 9), _random(30_000, 30_000, 36)))),
    # nearly every bucket huge; all of them (the full sort of all entries)
    "dense": (70, *_random(70, 1_146_000, 37)),
    "dense_over": (70, *_random(70, 1_200_000, 38)),
}


@pytest.mark.parametrize("name", list(HUGE_CASES))
def test_huge_buckets_equal_oracle(name):
    import paper_2509_02590_gb300 as wcc
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    n, u, v = HUGE_CASES[name]
    for seed in (None, 1):  # as they are, and shuffled
        p = np.arange(len(u)) if seed is None else np.random.default_rng(seed).permutation(len(u))
        src, dst = u[p].astype(np.int32), v[p].astype(np.int32)
        off, adj = oracle.build_csr(n, src, dst)
        with wcc.WccGraph.from_edges(torch.from_numpy(src).cuda(), torch.from_numpy(dst).cuda(), n) as g:
            goff, gadj = g.csr()
        assert np.array_equal(goff, off) and np.array_equal(gadj, adj)


@pytest.mark.parametrize("n", [64 * (2**20 - 1), 64 * (2**20 - 1) + 1])
def test_most_buckets_and_one_more_row(n):
    """Just under 2^26 rows there are 2^20 - 1 buckets of 64 rows, the most; from
    the next row on all entries are sorted at once."""
    import paper_2509_02590_gb300 as wcc
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    u, v = _random(n, 200_000, 40)
    u[:5], v[:5] = [n - 1, n - 2, n - 1, 0, n - 65], [n - 2, n - 1, 0, n - 1, n - 1]
    u[5:3000] = n - 1 - u[5:3000] % 130  # the last buckets are not empty
    src, dst = u.astype(np.int32), v.astype(np.int32)
    off, adj = oracle.build_csr(n, src, dst)
    with wcc.WccGraph.from_edges(torch.from_numpy(src).cuda(), torch.from_numpy(dst).cuda(), n) as g:
        goff, gadj = g.csr()
    assert np.array_equal(goff, off) and np.array_equal(gadj, adj)


def _copies_of_one_edge(extra):
    """2^30 + extra edges on 900,000 vertices, all but 5,000 of them 0-1: more
    than 2^31 entries in the first bucket, which holds rows 0 and 1.  Run in a
    process of its own, whose device memory (about 130 GB) goes with it."""
    import paper_2509_02590_gb300 as wcc
    n, m, k = 900_000, 2**30 + extra, 5000
    u, v = _random(n, k, 30)
    src = torch.zeros(m, dtype=torch.int32, device="cuda")
    dst = torch.ones(m, dtype=torch.int32, device="cuda")
    src[7:7 + k] = torch.from_numpy(u.astype(np.int32)).cuda()
    dst[7:7 + k] = torch.from_numpy(v.astype(np.int32)).cuda()
    off, adj = oracle.build_csr(n, np.append(u, 0).astype(np.int32), np.append(v, 1).astype(np.int32))
    with wcc.WccGraph.from_edges(src, dst, n) as g:
        goff, gadj = g.csr()
    assert np.array_equal(goff, off) and np.array_equal(gadj, adj)


def test_bucket_of_more_than_2_31_entries():
    import os
    import subprocess
    import sys
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    if torch.cuda.mem_get_info()[0] < 160 << 30:
        pytest.skip("needs 160 GB of free device memory")
    code = "import tests.test_gpu_csr_buckets as t; t._copies_of_one_edge(10_000)"
    subprocess.run([sys.executable, "-c", code], check=True, timeout=300,
                   cwd=os.path.dirname(os.path.dirname(os.path.abspath(__file__))))
