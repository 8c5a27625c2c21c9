"""Bottom-node products by packed row gathers (kernels_bh.cu) against the
oracle, at the widths where the kernel's tiles change: a one-column root
without environment operators, sectors of a few columns (32-row tiles shared
by the warps of a CTA), the first widths past that (16-row tiles), and sectors
wider than a warp; every charge sector's last tile is ragged."""
import numpy as np
import pytest

from oracle import model as omodel, ttn as ottn

from ttn_layout import from_layout, to_layout

pytestmark = pytest.mark.gpu

KW = dict(t=1.0, m=0.7, ge2=1.0, cB=0.5, nu=10.0)


@pytest.fixture(scope="module")
def q():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_2011_10658_gb300 as pkg
    pkg.lib()
    return pkg


@pytest.mark.parametrize("L,chi,Q", [((2, 1, 1), 8, 0), ((2, 2, 1), 3, 1), ((2, 2, 1), 24, 0), ((2, 2, 1), 31, 2),
                                     ((2, 2, 1), 70, 0)])
def test_product_and_adjoint_equal_oracle(q, L, chi, Q):
    import torch
    ref = ottn.TTN(omodel.Params(*L, Q=Q, **KW), chi, 5)
    s = q.TTN(q.Model(*L, Q=Q, **KW), chi, seed=5, precision="fp64")
    ref.move_to(0)
    s.move_center(0)
    n = s.node_size(0)
    x = np.random.default_rng(2).standard_normal(n)
    want = to_layout(ref.heff_apply(0, from_layout(x, ref.labels[0], ref.T[0].shape)), ref.labels[0])
    xd = torch.from_numpy(x).cuda()
    yd = torch.full_like(xd, float("nan"))
    torch.cuda.synchronize()
    for call in (s.apply_heff_device, s.apply_heff_adjoint_device):
        call(xd.data_ptr(), yd.data_ptr(), n)
        torch.cuda.synchronize()
        assert np.max(np.abs(yd.cpu().numpy() - want)) < 1e-12 * np.max(np.abs(want))
        yd.fill_(float("nan"))


@pytest.mark.parametrize("chi", [3, 24, 31])
def test_correction_product_is_fp64_accurate(q, chi):
    """The residual a mixed update ends with, formed in FP64: the solver's own
    1e-10 |E| plus the float-float product's rounding (about sqrt(2500) 2^-44
    of an operator norm of a few hundred, 1.2e-9)."""
    s = q.TTN(q.Model(2, 2, 1, Q=0, **KW), chi, seed=5, precision="tf32x3")
    e = s.optimize_node(0, tol=1e-10, max_krylov=64)
    v = s.node_export(0)
    s.set_precision("fp64")
    assert np.linalg.norm(s.apply_heff(v) - e * v) < 1e-10 * abs(e) + 1.2e-9
