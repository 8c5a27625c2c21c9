"""Tensor-core upper-node products (grouped leg contractions) against the FP64
path: sectors of one column to past three MMA widths, trees where groups fill
and where they do not, and a product written over its own input."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

KW = dict(t=1.0, m=0.7, ge2=1.0, cB=0.5, nu=10.0)
# operand rounding of one product (two or three contractions in a row): BF16
# 2^-8, TF32 2^-11, three-product split 2^-21 with FP32 accumulation
TOL = {"bf16": 2e-2, "tf32": 3e-3, "tf32x3": 2e-5}


@pytest.fixture(scope="module")
def q():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_2011_10658_gb300 as pkg
    pkg.lib()
    return pkg


@pytest.mark.parametrize("L,chi,Q", [((4, 2, 2), 5, 1), ((4, 2, 2), 40, 0), ((4, 2, 2), 100, 2), ((4, 4, 2), 33, 0)])
def test_products_at_every_layer(q, L, chi, Q):
    import torch
    model = q.Model(*L, Q=Q, **KW)
    s = q.TTN(model, chi, seed=6, precision="fp64")
    tree = model.tree()
    for layer in range(1, tree[:, 0].max() + 1):
        node = int(np.nonzero(tree[:, 0] == layer)[0][-1])
        s.set_precision("fp64")
        s.move_center(node)
        x = np.random.default_rng(node).standard_normal(s.node_size(node))
        want = s.apply_heff(x)
        for precision in ("bf16", "tf32", "tf32x3"):
            s.set_precision(precision)
            y = s.apply_heff(x)
            err = np.max(np.abs(y - want)) / np.max(np.abs(want))
            assert err < TOL[precision], (node, precision, err)
            xd = torch.from_numpy(x).cuda()
            torch.cuda.synchronize()
            s.apply_heff_device(xd.data_ptr(), xd.data_ptr(), x.size)
            torch.cuda.synchronize()
            assert np.array_equal(xd.cpu().numpy(), y)
    s.close()
