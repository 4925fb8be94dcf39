"""Whole replicates per block: after an error of one of its units a block runs
no external transfer of that day, so the statistics of a failed run count the
day's other events only."""
import numpy as np
import pytest

from paper_1605_01421_gb300 import workloads as W

pytestmark = pytest.mark.gpu

N = 300


def _events(bad_exit, n_rep):
    """Days 1 and 2: ten exits and five transfers; on day 2, with bad_exit,
    node 7 also sends away more than it holds."""
    cols = []
    for day in (1, 2):
        cols += [(W.EXIT, day, 20 + i, 0, 1) for i in range(10)]
        cols += [(W.EXTERNAL, day, 100 + i, 200 + i, 2) for i in range(5)]
    if bad_exit:
        cols.append((W.EXIT, 2, 7, 0, 1000))
    kind, t, node, dest, n = (np.array(c, np.int32) for c in zip(*cols))
    m = t.size
    return dict(event=kind, time=t, node=node, dest=dest, n=n, proportion=np.zeros(m),
                select=np.full(m, 2, np.int32), shift=np.full(m, -1, np.int32))


@pytest.mark.parametrize("fault", ["event", "rate"])
@pytest.mark.parametrize("graphs", [False, True])
def test_no_transfers_after_an_error_of_the_day(fault, graphs):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1605_01421_gb300 import binding
    v0 = np.full((N, 1), 0.2)
    if fault == "rate":
        v0[9] = -1.0  # a negative rate on day 1
    w = W.plain_model(W.SISE, np.tile([[40, 2]], (N, 1)), np.arange(0, 5), W.sise_gdata(), seed=2,
                      v0=v0, events=_events(fault == "event", 1))
    m = binding.Model(w)
    m.set_tuning(N, 4)
    m.set_graphs(graphs)
    dev = lambda a, t: torch.as_tensor(np.ascontiguousarray(a, t), device="cuda")  # noqa: E731
    U = torch.empty((1, 5, N, 2), dtype=torch.int32, device="cuda")
    V = torch.empty((1, 5, N, 1), dtype=torch.float64, device="cuda")
    rc, st, er = m.run(w.tspan, w.seed, 1, dev(w.u0, np.int32), dev(w.v0, np.float64), U, V,
                       stream=torch.cuda.Stream(), check=False)
    m.close()
    if fault == "event":
        assert (rc, er["node"], er["day"]) == (-2, 7, 2)
        assert st["events_applied"] == 15 + 10
    else:
        assert (rc, er["node"], er["day"]) == (-4, 9, 1)
        assert st["events_applied"] == 10
