"""A forced tile shape (QED_KC_SHAPE) takes bottom-node FP64 products to the
dense grouped kernel as well, where it checks the packed row gathers: with
couplings that are no powers of two the two kernels scale different operands
by a term's coefficient, so the results agree to rounding and not to the bit."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

KW = dict(t=0.9, m=0.7, ge2=1.1, cB=0.35, nu=10.3, Q=0)


@pytest.mark.parametrize("shape", ["16", "64", "1664"])
def test_dense_product_checks_the_gathers(shape, monkeypatch):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_2011_10658_gb300 as q
    y = []
    for forced in (None, shape):
        if forced:
            monkeypatch.setenv("QED_KC_SHAPE", forced)
        s = q.TTN(q.Model(2, 2, 1, **KW), 12, seed=3, precision="fp64")
        s.move_center(0)
        x = np.random.default_rng(1).random(s.node_size(0)) - 0.5
        y.append(s.apply_heff(x))
        s.close()
    assert np.max(np.abs(y[0] - y[1])) < 1e-12 * np.max(np.abs(y[0]))
    assert not np.array_equal(y[0], y[1])
