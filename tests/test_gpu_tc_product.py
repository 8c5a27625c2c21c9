"""Tensor-core bottom-node products against the FP64 path at the widths where
the gather kernel changes: rows of 2 to 16 sixteen-byte pieces (those without a
specialisation among them), ragged last tiles, terms that reach only some of a
tile's rows, and a state switched between operand formats."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

KW = dict(t=1.0, m=0.7, ge2=1.0, cB=0.5, nu=10.0)
# operand rounding of one product: unit roundoff 2^-8, 2^-11; three-product
# split 2^-21 with FP32 accumulation
TOL = {"bf16": 2e-2, "tf32": 3e-3, "tf32x3": 2e-5}


@pytest.fixture(scope="module")
def q():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_2011_10658_gb300 as pkg
    pkg.lib()
    return pkg


@pytest.mark.parametrize("L,chi,Q", [((2, 2, 1), 12, 0), ((2, 2, 1), 50, 1), ((2, 2, 1), 80, 0), ((2, 2, 1), 115, 0),
                                     ((4, 2, 2), 20, 2)])
def test_products_in_every_format(q, L, chi, Q):
    model = q.Model(*L, Q=Q, **KW)
    s = q.TTN(model, chi, seed=6, precision="fp64")
    for node in (0, 1):
        s.set_precision("fp64")
        s.move_center(node)
        x = np.random.default_rng(node).standard_normal(s.node_size(node))
        want = s.apply_heff(x)
        for precision in ("bf16", "tf32", "tf32x3", "bf16"):
            s.set_precision(precision)
            if precision == "tf32x3" and max(model.sectors(chi)[node].values()) > 64:
                # its two stages of hi and lo rows exceed an SM's shared memory
                with pytest.raises(q.QedError) as refused:
                    s.apply_heff(x)
                assert refused.value.code == -7
                continue
            err = np.max(np.abs(s.apply_heff(x) - want)) / np.max(np.abs(want))
            assert err < TOL[precision], (node, precision, err)
    s.close()
