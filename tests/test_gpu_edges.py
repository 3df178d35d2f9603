"""Sizes at which a kernel's split of the work changes, against the oracle: the triangle listing's
windows and its light / heavy boundary (cliques), rows of a few communities at the degree limits of
a warp and of a CTA, removals and validation at the edges of 32-entry words and of a warp's chunk."""
import numpy as np
import pytest

import graphgen
import oracle
from tests.conftest import csr_from_edges

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def rs():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2508_01485_gb300 as rsgpu
    return rsgpu


def _check(G, off, cols, labels, k):
    s, wmax = G.score(want_omega_max=True)
    assert G.device_errors() == 0
    o = oracle.Oracle(off, cols, labels, k)
    assert abs(wmax - o.wmax) <= 1e-12 * o.wmax
    np.testing.assert_allclose(s.cpu().numpy(), o.scores(), rtol=1e-12, atol=0)


@pytest.mark.parametrize("mirror", [1, 0])
@pytest.mark.parametrize("k", [200, 7])
@pytest.mark.parametrize("m", [3, 33, 128, 129, 130, 200])
def test_cliques(rs, m, k, mirror):
    """A clique of m nodes among isolated ones: out-degrees m - 1 .. 0 in G_x with a community
    each, so windows that end at 128 entries, nodes with 127 to 129 out-neighbours, and every pair
    closing a triangle (each entry's sums at their largest)."""
    rng = np.random.default_rng(m)
    at = np.sort(rng.choice(3 * m, m, replace=False))
    off, cols = csr_from_edges(3 * m, [(int(a), int(b)) for i, a in enumerate(at) for b in at[:i]])
    labels = rng.integers(0, k, 3 * m).astype(np.int32)
    labels[at] = rng.permutation(m) % k
    G = rs.Graph.build(off, cols, labels, k)
    G.set_tuning(p3_mirror=mirror)
    _check(G, off, cols, labels, k)


@pytest.mark.parametrize("d", [32, 33, 511, 512, 513, 16384, 16385])
def test_long_rows_of_few_communities(rs, d):
    """Two joined centres with d neighbours each in three communities: the table is small at any
    degree, so the degree alone decides between a warp, a CTA and the hub path."""
    n = 2 + d + 40
    rng = np.random.default_rng(d)
    edges = [(0, 1)] + [(0, 2 + i) for i in range(d - 1)] + [(1, n - 1 - i) for i in range(d - 1)]
    edges += [(int(a), int(b)) for a, b in rng.integers(2, n, (2 * d, 2))]
    off, cols = csr_from_edges(n, edges)
    labels = rng.integers(0, 3, n).astype(np.int32)
    labels[:2] = 0, 1
    _check(rs.Graph.build(off, cols, labels, 3), off, cols, labels, 3)


@pytest.mark.parametrize("m", [31, 32, 33, 64, 200])
def test_removals_at_word_edges(rs, m):
    """Compaction over words of 32 entries: sizes at their edges, runs of dead words, everything
    removed, and a second removal on the compacted graph."""
    rng = np.random.default_rng(m)
    edges = {(int(min(a, b)), int(max(a, b))) for a, b in rng.integers(0, m, (4 * m, 2)) if a != b}
    off, cols = csr_from_edges(m, sorted(edges))
    labels = rng.integers(0, 5, m).astype(np.int32)
    G = rs.Graph.build(off, cols, labels, 5)
    gone = []
    for step in (rng.permutation(m)[: m // 8], np.arange(m // 2), np.arange(m)):
        cut = list(rng.permutation(sorted(edges))[:5])
        G.apply_removals(step, [tuple(map(int, e)) for e in cut])
        gone.extend(int(v) for v in step)
        edges = {e for e in edges if e[0] not in gone and e[1] not in gone and list(e) not in [list(map(int, c)) for c in cut]}
        off, cols = csr_from_edges(m, sorted(edges))
        s = G.score().cpu().numpy()
        np.testing.assert_allclose(s, oracle.Oracle(off, cols, labels, 5).scores(), rtol=1e-12, atol=0)


@pytest.mark.parametrize("gap", [0, 33, 5000])
@pytest.mark.parametrize("at", [0, 1, 511, 512, 513, 1023, -1])
def test_validation_at_chunk_edges(rs, gap, at):
    """One entry re-pointed at the edges of a warp's 512 entries, with runs of isolated nodes
    between the rows: found whatever the place; the untouched graph passes."""
    rng = np.random.default_rng(7)
    m = 60
    n = m * (gap + 1)
    node = np.arange(m) * (gap + 1) + gap
    pairs = [(int(node[i]), int(node[j])) for i in range(m) for j in range(i) if rng.random() < 0.5]
    off, cols = csr_from_edges(n, pairs)
    labels = np.zeros(n, np.int32)
    rs.Graph.build(off, cols, labels, 2).close()
    bad = cols.copy()
    row = int(np.searchsorted(off, at % len(cols), side="right")) - 1
    others = np.setdiff1d(np.arange(n)[gap:gap + 100 * (gap + 1)], np.append(cols[off[row]:off[row + 1]], row))
    bad[at] = others[np.abs(others.astype(np.int64) - int(bad[at])).argmin()]
    with pytest.raises(rs.RSError) as e:
        rs.Graph.build(off, bad, labels, 2)
    assert e.value.status == rs.RS_EINVAL
    unsorted = cols.copy()
    if off[row + 1] - off[row] >= 2:
        a = int(off[row])
        unsorted[a], unsorted[a + 1] = unsorted[a + 1], unsorted[a]
        with pytest.raises(rs.RSError):
            rs.Graph.build(off, unsorted, labels, 2)
    labels[n - 1] = 2
    with pytest.raises(rs.RSError):
        rs.Graph.build(off, cols, labels, 2)


@pytest.mark.parametrize("removed", [1, 40, 400])
def test_whatif_with_few_and_many_pairs_per_warp(rs, removed):
    """The triangle search takes one pair of a touched node and a neighbour per warp, or many:
    the same bits as a full rescoring."""
    g = graphgen.dcsbm_small(50000, seed=8, dmax=3000, mu=0.4)
    nodes = np.random.default_rng(removed).choice(g.n, removed, replace=False)
    srv = rs.Server([rs.Graph.from_generated(g)], max_slots=1, max_top_k=10)
    a, path = srv.whatif(0, nodes=nodes, full="incremental")
    b, _ = srv.whatif(0, nodes=nodes, full=True)
    assert path == 1
    np.testing.assert_array_equal(a.cpu().numpy().view(np.uint64), b.cpu().numpy().view(np.uint64))
    srv.close()


def test_full_request_needs_no_second_poll_to_run(rs):
    """A poll that admits full requests leaves all of their work in the device's queues."""
    g = graphgen.sbm_2000()
    srv = rs.Server([rs.Graph.from_generated(g)], max_slots=3, max_top_k=10, mode="full")
    for i in range(3):
        srv.submit(0, nodes=[i], edges=[], top_k=10)
    done = list(srv.poll(block=False))
    torch.cuda.synchronize()
    done += list(srv.poll(block=False))
    assert len(done) == 3 and all(status == 0 and path == 0 for _, status, path, _, _ in done)
    srv.close()
