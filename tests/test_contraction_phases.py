"""Contraction passes grown phase by phase.

A capped maximum-adjacency pass merges exactly its phases: a pick of largest
key below the cap (ties to the smallest id) and the closure after it, every
vertex that gets cap edges into the added set, in whatever order the closure
is grown.  The CPU test checks that claim against the sequential pass
(tests/_helpers.py), first pass and later ones; the GPU test compares the
kernel, which grows the closures with the whole block, with the oracle at
the sizes where its loops change form.
"""
import numpy as np
import pytest

import oracle
import synth
from tests._helpers import contract_passes


def _phases(n, eu, ev, rep, k, rng):
    """One pass on the sets rep, each closure grown in a random order."""
    roots = np.unique(rep)
    w = {int(a): {} for a in roots}
    for x, y in zip(rep[eu], rep[ev]):
        if x != y:
            w[int(x)][int(y)] = w[int(x)].get(int(y), 0) + 1
            w[int(y)][int(x)] = w[int(y)].get(int(x), 0) + 1
    key = {int(a): 0 for a in roots}
    out = rep.copy()
    while key:
        first = min(key, key=lambda a: (-key[a], a))
        phase, todo = [first], [first]
        del key[first]
        while todo:
            x = todo.pop(int(rng.integers(0, len(todo))))
            for y, c in w[x].items():
                if y in key:
                    key[y] += c
                    if key[y] >= k:
                        del key[y]
                        phase.append(y)
                        todo.append(y)
        out[np.isin(rep, phase)] = min(phase)
    return out


@pytest.mark.parametrize("k", [1, 2, 3, 4, 6])
def test_phases_equal_the_sequential_passes(k):
    rng = np.random.default_rng(40 + k)
    merged = several = 0
    for _ in range(60):
        n = int(rng.integers(2, 40))
        eu, ev = synth.random_gnp(n, float(rng.uniform(0.05, 0.6)), rng)
        if len(eu) == 0:
            continue
        rep, passes = np.arange(n), 0
        while len(np.unique(rep)) > 1:
            new = _phases(n, eu, ev, rep, k, rng)
            passes += 1
            if np.array_equal(new, rep):
                break
            rep = new
        ref, ref_passes = contract_passes(n, eu, ev, k)
        assert np.array_equal(rep, ref) and passes == ref_passes
        merged += len(np.unique(rep)) < n
        several += passes > 1
    assert merged >= 10 and several >= 10


def _clusters(sizes, seed):
    """One cluster of each size, of one of four kinds: sparse random, dense
    random, two random halves joined by one to three edges, and a hub joined
    to everything over a sparse rest (rows longer than any other)."""
    rng = np.random.default_rng(seed)
    eu, ev, lab, base = [], [], [], 0
    for c, s in enumerate(sizes):
        kind = c % 4
        if kind == 2 and s >= 12:
            h = s // 2
            for lo, hi in ((0, h), (h, s)):
                a, b = synth.random_gnp(hi - lo, min(1.0, 9.0 / (hi - lo)), rng)
                eu.append(base + lo + a), ev.append(base + lo + b)
            j = int(rng.integers(1, 4))
            eu.append(base + rng.integers(0, h, j)), ev.append(base + rng.integers(h, s, j))
        else:
            mean = (4.5, 14.0, 14.0, 5.0)[kind]
            a, b = synth.random_gnp(s, min(1.0, mean / s), rng)
            eu.append(base + a), ev.append(base + b)
            if kind == 3:
                eu.append(np.full(s - 1, base)), ev.append(base + np.arange(1, s))
        lab.append(np.full(s, c))
        base += s
    perm = rng.permutation(base)
    s, d = synth.graphs._dedup(base, perm[np.concatenate(eu)], perm[np.concatenate(ev)])
    labels = np.empty(base, np.int32)
    labels[perm] = np.concatenate(lab)
    return synth.Workload("clusters", base, s, d, labels, 2)


EDGES = [2, 3, 9, 10, 11, 31, 32, 33, 63, 64, 65, 66, 67, 97, 127, 128, 129, 130, 191, 255, 256,
         257, 258, 383, 511, 512, 513, 514, 700, 1023, 1024, 1025, 1026]
RULES = {"log10": oracle.RULE_LOG10, "log2": oracle.RULE_LOG2, "sqrt": oracle.RULE_SQRT}


@pytest.mark.gpu
@pytest.mark.parametrize("rule", list(RULES))
@pytest.mark.parametrize("env", [{}, {"WCC_TINY_N": "0"}, {"WCC_DENSE_NSV": "0", "WCC_TINY_N": "0"},
                                 {"WCC_SMEM_KB": "16", "WCC_DENSE_NSV": "3"}])
def test_refinement_at_loop_edges(monkeypatch, rule, env):
    torch = pytest.importorskip("torch")
    import paper_2509_02590_gb300 as wcc
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    for k, v in env.items():
        monkeypatch.setenv(k, v)
    # every kind at every size: the sizes in four rotations
    for turn in range(4):
        w = _clusters(EDGES[turn:] + EDGES[:turn], 100 + turn)
        off, adj = oracle.build_csr(w.n, w.src, w.dst)
        ref, _ = oracle.wcc(w.n, off, adj, w.labels, w.min_size, kind=RULES[rule])
        with wcc.WccGraph.from_edges(w.src, w.dst, w.n) as g:
            out, st = g.run(w.labels, min_size=w.min_size, rule=rule, stats=True)
        assert np.array_equal(out, ref), (turn, rule, env)
        assert st["out_clusters"] == int(ref.max(initial=-1)) + 1


@pytest.mark.gpu
@pytest.mark.parametrize("env", [{}, {"WCC_TINY_N": "0", "WCC_SMEM_KB": "16"}])
def test_components_of_long_thin_clusters(monkeypatch, env):
    """Clusters of paths, whose components take as many rounds to grow as the
    paths are long: around the rounds after which the union-find takes over, in
    one path and summed over several, and far beyond; after a star of 1,100
    leaves, which a round adds at once, only after as many more.  With T = 0 the
    components are the output."""
    torch = pytest.importorskip("torch")
    import paper_2509_02590_gb300 as wcc
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    for k, v in env.items():
        monkeypatch.setenv(k, v)
    clusters = [[L] for L in (32, 33, 34, 35, 64, 65, 66, 67, 129, 1000, 5000)]
    clusters += [[33, 33], [33, 34], [17, 17, 17], [2, 65], [65, 2], [3, 2000, 1], [2] * 40]
    clusters += [[-1100, L] for L in (30, 34, 35, 36, 70)]  # -k: a star of k leaves
    for shuffled in (False, True):
        eu, ev, lab, base = [], [], [], 0
        for c, paths in enumerate(clusters):
            for L in paths:
                size = L if L > 0 else 1 - L
                eu.append(base + (np.arange(L - 1) if L > 0 else np.zeros(-L, np.int64)))
                ev.append(base + np.arange(1, size))
                lab.append(np.full(size, c))
                base += size
        perm = np.random.default_rng(1).permutation(base) if shuffled else np.arange(base)
        s, d = synth.graphs._dedup(base, perm[np.concatenate(eu)], perm[np.concatenate(ev)])
        labels = np.empty(base, np.int32)
        labels[perm] = np.concatenate(lab)
        off, adj = oracle.build_csr(base, s, d)
        ref, _ = oracle.wcc(base, off, adj, labels, 2, kind=oracle.RULE_LINEAR, num=0, den=1)
        assert ref.max() + 1 == sum(abs(L) > 1 for paths in clusters for L in paths)
        with wcc.WccGraph.from_edges(s, d, base) as g:
            out = g.run(labels, min_size=2, rule="linear", num=0, den=1)
        assert np.array_equal(out, ref)
