"""Basis lengths around the eight columns of a dot sweep, whether or not a run
gets to its tolerance in them: the energy returned is the Ritz value of the
tensor written, and its residual is what the solver reports."""
import ctypes

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

KW = dict(t=1.0, m=0.7, ge2=1.0, cB=0.5, nu=10.0, Q=0)


@pytest.fixture(scope="module")
def q():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_2011_10658_gb300 as pkg
    pkg.lib()
    return pkg


@pytest.mark.parametrize("precision", ["fp64", "tf32x3"])
@pytest.mark.parametrize("L,chi,node", [((4, 2, 2), 12, 14), ((4, 2, 2), 16, 8), ((2, 2, 1), 16, 0)])
def test_ritz_pair_of_short_bases(q, L, chi, node, precision):
    """The reported residual |beta s| is exact up to the loss of orthogonality
    (1e-12) and rounding, the bounds of test_gpu_lanczos_step.py: 1.4e-11 in
    FP64, 3e-9 with the float-float products of a mixed state."""
    from paper_2011_10658_gb300._lib import check, lib
    floor = 1.4e-11 if precision == "fp64" else 3e-9
    s = q.TTN(q.Model(*L, **KW), chi, seed=2, precision=precision)
    s.move_center(node)
    start = s.node_export(node)
    for krylov in (7, 8, 9, 15, 16, 17):
        s.node_import(node, start)
        e = ctypes.c_double()
        check(lib().ttn_optimize_node(s._h, node, 1e-6, krylov, ctypes.byref(e)), allow=(-4,))
        u = s.last_update()
        v = s.node_export(node)
        s.set_precision("fp64")
        hv = s.apply_heff(v)
        s.set_precision(precision)
        assert abs(np.linalg.norm(v) - 1.0) < 1e-13
        assert abs(v @ hv - e.value) < 1e-12 * abs(e.value) + floor
        assert abs(np.linalg.norm(hv - e.value * v) - u["rel_residual"] * abs(e.value)) < 1e-3 * u["rel_residual"] * abs(e.value) + floor
    s.close()
