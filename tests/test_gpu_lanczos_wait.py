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


def test_batch_member_that_times_out(q):
    """One member's failure ends the call; no member is left on its
    reduced-precision operator (the gradient of the second one is what an FP64
    state with its tensors has, up to the operators' 1e-11; 1e-6 apart otherwise)."""
    import torch
    stream = torch.cuda.current_stream().cuda_stream
    model = q.Model(2, 2, 2, **KW)
    pair = [q.TTN(model, 8, seed=i, precision="tf32x3", stream=stream) for i in (1, 2)]
    pair[0].set_wait_limit(0)
    with pytest.raises(q.QedError) as ei:
        q.batch_sweep(pair, 1, tol=1e-6, max_krylov=16)
    assert ei.value.code == -6
    s = pair[1]
    s.move_center(s.info()["n_nodes"] - 1)
    r = q.TTN(model, 8, seed=2, precision="fp64", stream=stream)
    r.load_tensors([s.node_export(i) for i in range(s.info()["n_nodes"])])
    node = 0
    got = []
    for t in (s, r):
        t.move_center(node)
        x = torch.from_numpy(np.random.default_rng(3).random(t.node_size(node)) - 0.5).cuda()
        y = torch.empty_like(x)
        t.energy_grad_device(node, x.data_ptr(), y.data_ptr(), x.numel())
        torch.cuda.synchronize()
        got.append(y.cpu().numpy())
    assert np.linalg.norm(got[0] - got[1]) < 1e-9 * np.linalg.norm(got[1])
    pair[0].set_wait_limit(-1)
    q.batch_sweep(pair, 1, tol=1e-6, max_krylov=16)
    for t in pair + [r]:
        t.close()
