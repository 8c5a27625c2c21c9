"""A grid barrier of the one-launch Lanczos step that runs out: the wait bound
is zero polls, so every barrier gives up at once; the step goes on in bounds,
marks the run as failed and returns.  The update reports QED_ETIMEOUT, the node
keeps its tensor, and with the default bound the same update is what a fresh
state's is."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

KW = dict(t=1.0, m=1.0, ge2=1.0, cB=0.5, nu=10.0, Q=0)


@pytest.fixture(scope="module")
def q():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_2011_10658_gb300 as pkg
    pkg.lib()
    return pkg


# the short form (n <= 16384) and the long one, several blocks each
@pytest.mark.parametrize("L,chi,node", [((4, 2, 2), 16, 12), ((2, 2, 2), 16, 0)])
def test_timeout_keeps_the_tensor(q, L, chi, node):
    def fresh():
        s = q.TTN(q.Model(*L, **KW), chi, seed=6, precision="fp64")
        s.move_center(node)
        return s

    s = fresh()
    start = s.node_export(node)
    s.set_wait_limit(0)
    with pytest.raises(q.QedError) as ei:
        s.optimize_node(node, tol=1e-8)
    assert ei.value.code == -6
    np.testing.assert_array_equal(s.node_export(node), start)
    s.set_wait_limit(-1)
    e = s.optimize_node(node, tol=1e-8)
    r = fresh()
    want = r.optimize_node(node, tol=1e-8)
    assert abs(e - want) <= 1e-11 * abs(want)
    s.close()
    r.close()
