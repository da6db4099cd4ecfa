"""Breadth-first graph codes of the hull lookup (CPU only): from any directed
edge of a relabelled template triangulation the code is listed, and names exactly
the Weinberg start edges, with the labels and candidate list of the walk from
each."""
import numpy as np

from paper_1603_05143_gb300 import tables as T


def test_code_from_any_edge_names_the_weinberg_starts():
    *_, entries, _ = T.build()
    entry_of = {code: i for i, code in enumerate(sorted(entries))}
    graphs = T.graph_codes(entry_of)
    rng = np.random.default_rng(23)
    for S, name in enumerate(T.TEMPLATE_NAMES):
        k = T.K[S]
        tris = T.triangulations(T.normalised_template(name))
        for i in rng.permutation(len(tris))[:200]:
            new = rng.permutation(k)
            facets = [tuple(int(new[x - 1]) for x in np.roll(f, rng.integers(3))) for f in tris[i]]
            th = T._third(facets)
            edges = list(th)
            u, v = edges[rng.integers(len(edges))]
            order, code = T.breadth_first(th, k, u, v)
            assert sorted(order) == list(range(k))
            deg = {x: sum(x in f for f in facets) for x in range(k)}
            top = max(T.edge_key(deg, th, a, b) for a, b in edges)
            starts = {e for e in edges if T.edge_key(deg, th, *e) == top}
            if len(starts) == len(edges):
                starts = {(u, v)}
            listed = graphs[(k, code)]
            assert {(order[a], order[b]) for a, b, _, _ in listed} == starts, name
            for a, b, perm, ent in listed:
                wcode, lab = T.weinberg(facets, order[a], order[b])
                assert entry_of[wcode] == ent
                assert all(perm >> (4 * l) & 15 == lab[x] for l, x in enumerate(order))


def test_packed_rows_differ_for_different_codes():
    graphs = T.graph_codes({c: i for i, c in enumerate(sorted(T.build()[3]))})
    packed = {(k, tuple(T.pack_rows(rows))) for k, rows in graphs}
    assert len(packed) == len(graphs) and all(len(r) == 7 for _, r in packed)


def test_rank_in_the_start_rows_is_the_place_in_the_list():
    for (k, _), starts in T.graph_codes({c: i for i, c in enumerate(sorted(T.build()[3]))}).items():
        words = T.start_rows(starts)
        assert len(words) == 4 * T.TIE_HEAD
        bits = sum(w << (32 * i) for i, w in enumerate(words))
        assert bin(bits).count("1") == len(starts)
        for i, (u, v, *_) in enumerate(starts):
            at = 16 * u + v
            assert bits >> at & 1 and bin(bits & ((1 << at) - 1)).count("1") == i, k
