"""A day's external transfers in chains of dependent waves, large ones (32
individuals or more, sampled by warps) following small ones: every kernel
that runs them gives the oracle's trajectories."""
import numpy as np
import pytest

from paper_1605_01421_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _chains(n_nodes, n_rep, per_rep):
    """Days of 1, 2, 31, 32, 33 and 150 waves: node 0 sends to one node after
    the other, every third time 32 to 40 individuals, and, beside each wave,
    up to five nodes send to node 0's next destinations."""
    cols = []
    for r in range(n_rep if per_rep else 1):
        rng = np.random.default_rng(40 + r)
        for day, waves in enumerate([1, 2, 31, 32, 33, 150], start=1):
            for i in range(waves + r):
                size = int(rng.integers(32, 41)) if i % 3 == 2 else int(rng.integers(1, 6))
                cols.append((day, 0, 1 + (i * 7) % (n_nodes - 60), size, r))
            for i in range(5):
                cols.append((day, n_nodes - 50 + 8 * i + day, 1 + i, 33 - i, r))
    t, node, dest, n, rep = (np.array(c, np.int32) for c in zip(*cols))
    m = t.size
    ev = dict(event=np.full(m, W.EXTERNAL, np.int32), time=t, node=node, dest=dest, n=n,
              proportion=np.zeros(m), select=np.full(m, 2, np.int32),
              shift=np.full(m, -1, np.int32))
    if per_rep:
        ev["rep"] = rep
    return ev


@pytest.mark.parametrize("per_rep", [False, True])
@pytest.mark.parametrize("mode,nodes,tuning", [
    ("separate", 200, (64, 2)),      # E2 kernel, state in shared memory
    ("separate", 30000, (64, 2)),    # E2 kernel, state in device memory
    ("fused", 200, (64, 2)),         # last block of a replicate
    ("inblock", 200, (200, 2)),      # whole replicates per block
    ("inblock", 200, (400, 2)),
])
def test_chains_of_waves(orc, mode, nodes, tuning, per_rep):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1605_01421_gb300 import binding
    u0 = np.tile([[60, 4]], (nodes, 1))
    u0[0] = [9000, 400]
    w = W.plain_model(W.SISE, u0, np.arange(0, 8), W.sise_gdata(), seed=12, n_rep=2,
                      v0=np.full((nodes, 1), 0.4), events=_chains(nodes, 2, per_rep))
    code, U0, V0, R0, err = orc.run(w)
    assert code == 0, err
    m = binding.Model(w)
    m.set_fused_events(mode == "fused")
    m.set_tuning(*tuning)
    dev = lambda a, t: torch.as_tensor(np.ascontiguousarray(a, t), device="cuda")  # noqa: E731
    U = torch.empty(U0.shape, dtype=torch.int32, device="cuda")
    V = torch.empty(V0.shape, dtype=torch.float64, device="cuda")
    rc, st, er = m.run(w.tspan, w.seed, 2, dev(w.u0, np.int32), dev(w.v0, np.float64), U, V)
    m.close()
    assert rc == 0, er
    assert np.array_equal(U.cpu().numpy(), U0)
    assert np.array_equal(V.cpu().numpy().view(np.uint64), V0.view(np.uint64))
    assert st["events_applied"] == w.events["time"].size * (1 if per_rep else 2)
