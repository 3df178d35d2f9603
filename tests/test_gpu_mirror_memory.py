"""The G_x slots in 8 bytes (p3_mirror = 0) and in 16: the same bits, with hub rows found anew while
either layout is in place, and in a server's incremental and full paths."""
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


def _bits(t):
    return t.cpu().numpy().view(np.uint64)


@pytest.mark.parametrize("law", ["hubs", "small"])
def test_both_layouts_score_alike(rs, law):
    g = graphgen.dcsbm(30000, 3000, 5.0, 2.1, 4, 4000, 0.5, seed=45) if law == "hubs" else graphgen.sbm_2000()
    gone = np.argsort(-np.diff(g.offsets), kind="stable")[:50:7]
    scores = {}
    for mirror in (1, 0):
        G = rs.Graph.from_generated(g)
        G.set_tuning(p3_mirror=mirror)
        first = _bits(G.score())
        C = G.clone()                                     # classified with this layout in place
        C.set_tuning(warp_cap=64, cta_cap=64, hub_chunk=512)
        many_hubs = _bits(C.score())
        C.apply_removals(gone)
        scores[mirror] = first, many_hubs, _bits(C.score())
        assert G.device_errors() == 0 and C.device_errors() == 0
        G.set_tuning(p3_mirror=1 - mirror)
        np.testing.assert_array_equal(_bits(G.score()), first)
    for a, b in zip(scores[0], scores[1]):
        np.testing.assert_array_equal(a, b)
    np.testing.assert_array_equal(scores[0][0], scores[0][1])


def test_served_without_the_mirror_pass(rs):
    g = graphgen.dcsbm(30000, 3000, 5.0, 2.1, 4, 4000, 0.5, seed=45)
    G = rs.Graph.from_generated(g)
    G.set_tuning(p3_mirror=0)
    nodes = np.argsort(-np.diff(g.offsets), kind="stable")[3000:3004]
    srv = rs.Server([G], max_slots=1, max_top_k=10)
    a, path = srv.whatif(0, nodes=nodes, full="incremental")
    b, _ = srv.whatif(0, nodes=nodes, full=True)
    assert path == 1
    np.testing.assert_array_equal(_bits(a), _bits(b))
    srv.close()
