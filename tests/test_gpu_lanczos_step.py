"""The one-launch Lanczos step (kernels_lz.cu) through node updates, at the
sizes where its work split changes: nodes of a handful of rows (one block), a
few blocks, and more rows than the resident grid takes at once; basis lengths
around the eight columns of a dot sweep and the longest allowed; FP64 and
float-float arithmetic."""
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
def test_update_is_an_eigenpair_for_every_basis_length(q, L, chi, node, precision):
    """|H v - E v| is what the solver reports (tol |E|) plus the rounding of
    the check itself (64 eps of an operator norm below 1000, 1.4e-11; the
    float-float products of a mixed state 3e-9), and E does not depend on the
    basis length."""
    s = q.TTN(q.Model(*L, **KW), chi, seed=2, precision=precision)
    s.move_center(node)
    start = s.node_export(node)
    energies = []
    for krylov in (7, 8, 9, 17, 128):
        s.node_import(node, start)
        try:
            e = s.optimize_node(node, tol=1e-10, max_krylov=krylov)
        except q.QedError as err:   # 50 restarts of a short basis may not reach tol: the vector is valid all the same
            assert err.code == -4 and krylov < 17
            assert abs(np.linalg.norm(s.node_export(node)) - 1.0) < 1e-13
            continue
        v = s.node_export(node)
        assert abs(np.linalg.norm(v) - 1.0) < 1e-13
        s.set_precision("fp64")
        r = np.linalg.norm(s.apply_heff(v) - e * v)
        s.set_precision(precision)
        assert r < 1.01e-10 * abs(e) + (1.4e-11 if precision == "fp64" else 3e-9), (krylov, r)
        energies.append(e)
    assert np.ptp(energies) < 1e-9 * max(1.0, abs(energies[0]))
    s.close()
