"""Two states in two threads, each on a stream of its own: the Lanczos step is a
resident grid with barriers, and two of them (with everything else of an update)
share the GPU.  Every result is the one that the state gets alone, to the last
place (the tile shape is forced, because a tuned one is chosen by time)."""
import threading

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

KW = dict(t=1.0, m=1.0, ge2=1.0, cB=0.5, nu=10.0, Q=0)
JOBS = [((2, 2, 2), 16, "tf32x3", (0, 1, 4, 2, 6, 3)), ((4, 2, 2), 16, "fp64", (12, 8, 0, 1, 13, 14)),
        ((2, 2, 2), 12, "bf16", (3, 5, 2, 6, 0, 1))]


def run(q, torch, job, out):
    L, chi, precision, nodes = job
    try:
        stream = torch.cuda.Stream()
        s = q.TTN(q.Model(*L, **KW), chi, seed=7, precision=precision, stream=stream.cuda_stream)
        got = []
        for node in nodes:
            got.append(np.array([s.optimize_node(node, tol=1e-3, max_krylov=24)]))
            got.append(s.node_export(node))
        s.close()
        out.extend(got)
    except Exception as e:   # seen by the main thread
        out.append(e)


def test_threads_get_what_a_state_gets_alone(monkeypatch):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_2011_10658_gb300 as q
    q.lib()
    monkeypatch.setenv("QED_KC_SHAPE", "32")
    alone = [[] for _ in JOBS]
    for job, out in zip(JOBS, alone):
        run(q, torch, job, out)
    together = [[] for _ in JOBS]
    threads = [threading.Thread(target=run, args=(q, torch, job, out)) for job, out in zip(JOBS, together)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    for want, got in zip(alone, together):
        assert len(want) == len(got) == 12, [x for x in want + got if isinstance(x, Exception)]
        for a, b in zip(want, got):
            np.testing.assert_array_equal(a, b)
