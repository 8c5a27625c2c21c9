"""Two batched sweeps in one call do the same work as two calls: the second
visit to a node works on that visit's environment operators."""
import pytest

pytestmark = pytest.mark.gpu

KW = dict(t=1.0, m=0.7, ge2=1.0, cB=0.5, nu=10.0)


@pytest.mark.parametrize("precision", ["fp64", "tf32x3"])
def test_second_sweep_of_one_call_equals_a_second_call(precision):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_2011_10658_gb300 as q

    def states():
        return [q.TTN(q.Model(2, 2, 2, Q=0, **dict(KW, ge2=g)), 6, seed=3 + i, precision=precision)
                for i, g in enumerate((1.0, 2.0))]

    both = q.batch_sweep(states(), n=2, tol=1e-8, max_krylov=64)
    st = states()
    first = q.batch_sweep(st, n=1, tol=1e-8, max_krylov=64)
    second = q.batch_sweep(st, n=1, tol=1e-8, max_krylov=64)
    for b, x, y in zip(both, first, second):
        # eigenvalues to the solver's accuracy (tol squared over the gap, and
        # its drift through one sweep), the same products but for a few that
        # rounding moves across the tolerance
        assert abs(b["energy"] - y["energy"]) < 1e-7 * abs(y["energy"])
        assert abs(b["matvecs"] - x["matvecs"] - y["matvecs"]) <= 0.05 * (x["matvecs"] + y["matvecs"])
