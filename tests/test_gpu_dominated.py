"""Rows dominated by one community, joined in triangles: the directed values S of the Type-I terms are
small there (0.03 at 300,000 neighbours), and the scores have a closed form.

A centre x has d_x neighbours of its own community (leaves) and the two other centres of its triple,
each centre in a community of its own.  Leaving out one other centre's community, x's neighbours are
d_x + 1, one of them alone in its community: w = 2 H, H = log2(d + 1) - d log2(d) / (d + 1).  A centre's
only triads are the two of its triangle, so R(a) = S_b S_c (S_b + S_c) / (w_max D (D - 1)), S = w^(1/3),
D = d_a + 2; w_max = 2 (a centre's own column: its two cross neighbours in one community each)."""
import decimal

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _entropy(d):
    with decimal.localcontext(decimal.Context(prec=60)):
        d, two = decimal.Decimal(d), decimal.Decimal(2).ln()
        return (d + 1).ln() / two - d * d.ln() / two / (d + 1)


@pytest.mark.parametrize("mirror", [1, 0])
@pytest.mark.parametrize("degrees", [(20, 20, 20), (20, 300, 5000), (5000, 5000, 5000), (300, 20000, 300000), (300000, 300000, 20)])
def test_triangles_of_dominated_rows(degrees, mirror):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2508_01485_gb300 as rs
    first = 3 + np.cumsum([0, *degrees])
    n = int(first[-1])
    labels = np.repeat(np.arange(3), degrees).astype(np.int32)
    labels = np.concatenate([np.arange(3, dtype=np.int32), labels])
    # centres 0, 1, 2; leaf rows hold their centre alone
    rows = [np.concatenate([np.setdiff1d(np.arange(3), [x]), np.arange(first[x], first[x + 1])]) for x in range(3)]
    cols = np.concatenate([*rows, labels[3:]]).astype(np.int32)
    off = np.concatenate([[0], np.cumsum([len(r) for r in rows] + [1] * (n - 3))]).astype(np.int64)
    G = rs.Graph.build(off, cols, labels, 3)
    G.set_tuning(p3_mirror=mirror)
    got, wmax = G.score(want_omega_max=True)
    got = got.cpu().numpy()
    assert G.device_errors() == 0 and wmax == 2.0 and not got[3:].any()
    H = [_entropy(d) for d in degrees]
    with decimal.localcontext(decimal.Context(prec=60)):
        S = [(2 * h) ** (decimal.Decimal(1) / 3) for h in H]
        for a in range(3):
            b, c = (a + 1) % 3, (a + 2) % 3
            D = degrees[a] + 2
            want = S[b] * S[c] * (S[b] + S[c]) / (2 * D * (D - 1))
            # three cube roots of a quotient, a Newton step from a single-precision root each (2^-45),
            # and the log table's rounding, 2^-58 of an entropy H, of which a third reaches S
            tol = decimal.Decimal(2) ** -43 + decimal.Decimal(2) ** -58 * (1 / H[b] + 1 / H[c])
            assert abs(decimal.Decimal(float(got[a])) - want) <= tol * want, (a, float(got[a]), float(want))
