"""Batched sweeps in one call do the same work as one call each: a later visit to
a node works on that visit's environment operators (the grouped plans of the
first sweeps are rebuilt while buffers still grow or members finish early; one
problem's are kept in the fourth)."""
import pytest

pytestmark = pytest.mark.gpu

KW = dict(t=1.0, m=0.7, ge2=1.0, cB=0.5, nu=10.0)


@pytest.mark.parametrize("count", [1, 2])
@pytest.mark.parametrize("precision", ["fp64", "tf32x3"])
def test_sweeps_of_one_call_equal_single_calls(precision, count):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_2011_10658_gb300 as q

    def states():
        return [q.TTN(q.Model(2, 2, 2, Q=0, **dict(KW, ge2=g)), 6, seed=3 + i, precision=precision)
                for i, g in enumerate((1.0, 2.0)[:count])]

    together = q.batch_sweep(states(), n=4, tol=1e-8, max_krylov=64)
    st = states()
    single = [q.batch_sweep(st, n=1, tol=1e-8, max_krylov=64) for _ in range(4)]
    for i, b in enumerate(together):
        matvecs = sum(x[i]["matvecs"] for x in single)
        energy = single[-1][i]["energy"]
        # eigenvalues to the solver's accuracy (tol squared over the gap, and
        # its drift through one sweep), the same products but for a few that
        # rounding moves across the tolerance
        assert abs(b["energy"] - energy) < 1e-7 * abs(energy)
        assert abs(b["matvecs"] - matvecs) <= 0.05 * matvecs
