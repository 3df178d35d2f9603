"""Graphs whose hub lists and tables are kept from one change to the next: requests rescored on a
server's copies, removals, and scoring on a side stream give the bits of a graph built anew."""
import numpy as np
import pytest

import graphgen

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def rs():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2508_01485_gb300 as rsgpu
    return rsgpu


@pytest.fixture(scope="module")
def gen():
    return graphgen.dcsbm(30000, 3000, 5.0, 2.1, 4, 4000, 0.5, seed=45)


def _removals(g):
    """Node and edge lists that alternately keep the long rows and take most of them away."""
    by_degree = np.argsort(-np.diff(g.offsets), kind="stable")
    rng = np.random.default_rng(3)
    for i in range(10):
        nodes = by_degree[: 300 * (i // 2 + 1)] if i % 2 else rng.integers(0, g.n, i)
        v = rng.integers(0, g.n, 5)
        v = v[np.diff(g.offsets)[v] > 0]
        yield nodes, [(int(x), int(g.cols[g.offsets[x]])) for x in v]


def _bits(t):
    return t.cpu().numpy().view(np.uint64)


def _expected(rs, base, nodes, edges, k):
    G = base.clone()
    G.apply_removals(nodes, edges)
    off = G.score()
    ids, vals = G.topk(off, k)
    assert G.device_errors() == 0
    return ids.cpu().numpy(), _bits(vals), _bits(off)


@pytest.mark.parametrize("tuning", [{}, {"warp_cap": 64, "cta_cap": 64, "hub_chunk": 512}], ids=["few hubs", "many hubs"])
def test_more_full_requests_than_slots(rs, gen, tuning):
    base = rs.Graph.from_generated(gen)
    base.set_tuning(**tuning)
    reqs = list(_removals(gen))
    want = [_expected(rs, base, v, e, 100) for v, e in reqs]
    srv = rs.Server([base], max_slots=3, max_top_k=100, mode="full")
    tickets = {srv.submit(0, nodes=v, edges=e, top_k=100): i for i, (v, e) in enumerate(reqs)}
    while tickets:
        for ticket, status, path, ids, vals in srv.poll(block=True):
            i = tickets.pop(ticket)
            assert (status, path) == (0, 0)
            np.testing.assert_array_equal(ids, want[i][0])
            np.testing.assert_array_equal(vals.view(np.uint64), want[i][1])
    srv.close()


def test_removals_and_scores_on_a_side_stream(rs, gen):
    """Removal after removal on one graph, on a stream that does not wait for the legacy one."""
    side = torch.cuda.Stream()
    base = rs.Graph.from_generated(gen)
    G = base.clone()
    gone, cut = [], []
    out = torch.empty(gen.n, dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    for nodes, edges in _removals(gen):
        gone.extend(int(v) for v in nodes)
        cut.extend(edges)
        with torch.cuda.stream(side):
            G.apply_removals(nodes, edges)
            G.score_into(out)
        side.synchronize()
        np.testing.assert_array_equal(_bits(out), _expected(rs, base, gone, cut, 1)[2])
