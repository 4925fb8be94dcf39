"""Models of the built-in kinds with a caller's own S and G: the oracle's
trajectories where G keeps every rate current (draws decided from intervals),
where it leaves one stale (FP64 draw by draw), in threads and in warps, for
counts beyond the FP32 forms, and the same error where a count goes negative."""
import numpy as np
import pytest

from paper_1605_01421_gb300 import workloads as W

pytestmark = pytest.mark.gpu

_GDATA = {W.SIR: [0.5, 0.2], W.SIS: [0.003, 0.3], W.SISE: W.sise_gdata(),
          W.SISE_SP: W.sise_sp_gdata(), W.SISE3: W.sise3_gdata()}
# S (compartments x transitions) and the least G that keeps every rate current
_TABLES = {
    # a recovery adds two; an infected animal brings its own susceptible
    W.SIR: ([[-1, 1], [1, -1], [0, 2]], [[1, 1], [1, 1]]),
    # two new infected animals; recovered ones leave
    W.SIS: ([[-1, 0], [2, -1]], [[1, 1], [1, 1]]),
    W.SISE: ([[-1, 0], [1, -1]], [[1, 0], [1, 1]]),
    W.SISE_SP: ([[-1, 0], [1, -1]], [[1, 0], [1, 1]]),
}


def _tables(kind):
    if kind in _TABLES:
        return [np.array(t, np.int32) for t in _TABLES[kind]]
    # SISe3: recovered animals go to the next age class (the oldest leave)
    S, G = np.zeros((6, 6), np.int32), np.zeros((6, 6), np.int32)
    for a in range(3):
        S[2 * a, 2 * a], S[2 * a + 1, 2 * a] = -1, 1
        S[2 * a + 1, 2 * a + 1] = -1
        if a < 2:
            S[2 * a + 2, 2 * a + 1] = 1
    for j in range(6):
        for k in range(6):
            G[k, j] = S[k, j] != 0  # rate k reads compartment k
    return S, G


def _gpu():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1605_01421_gb300 import binding
    return binding


def _model(kind, herds, days, seed):
    rng = np.random.default_rng(seed)
    C = {W.SIR: 3, W.SISE3: 6}.get(kind, 2)
    u0 = np.stack([rng.integers(0, h, C) for h in herds])
    nv = 0 if kind in (W.SIR, W.SIS) else 1
    w = W.plain_model(kind, u0, np.arange(days + 1), _GDATA[kind], seed=seed, n_rep=2,
                      v0=rng.uniform(0, 2, (len(herds), nv)))
    w.S, w.G = _tables(kind)
    return w


def _same(orc, w, tuning=None):
    code, U0, V0, R0, err = orc.run(w)
    assert code == 0, err
    U1, V1, st = _gpu().simulate(w, tuning=tuning)
    assert np.array_equal(U0, U1)
    assert np.array_equal(V0.view(np.uint64), V1.view(np.uint64))
    assert st["reactions"] == int(R0.sum())


@pytest.mark.parametrize("kind", list(_GDATA))
@pytest.mark.parametrize("tuning", [None, (1, 1 << 20), (64, 3), (200, 2)])
def test_own_tables(orc, kind, tuning):
    herds = np.random.default_rng(kind).integers(1, 150, 301)
    herds[:5] = 900
    w = _model(kind, herds, 9, 30 + kind)
    _same(orc, w, tuning)
    w.G = np.ones_like(w.G)
    _same(orc, w, tuning)
    # the first transition leaves the last rate it changes stale
    w.G = _tables(kind)[1]
    w.G[np.flatnonzero(w.G[:, 0])[-1], 0] = 0
    _same(orc, w, tuning)


@pytest.mark.parametrize("own", [False, True])
@pytest.mark.parametrize("herd", [(1 << 20) + 3, (1 << 24) + 5, (1 << 30) + 7])
def test_large_counts(orc, own, herd):
    g = W.sise_gdata(gamma=2e3 / herd)
    w = W.plain_model(W.SISE, [[herd, herd], [herd, 40], [7, herd]], np.arange(3), g, seed=6,
                      v0=np.full((3, 1), 1e5 / herd))
    if own:
        w.S = np.array([[-1, 0], [3, -1]], np.int32)
    _same(orc, w)


@pytest.mark.parametrize("days_draws", [20000, 70000])
def test_days_of_many_draws(orc, days_draws):
    w = _model(W.SISE, [2, 2], 1, 8)
    w.u0[:] = [[40000, 40000], [39000, 41000]]
    w.gdata = np.asarray(W.sise_gdata(gamma=days_draws / 8e4))
    w.v0[:] = days_draws / 8e4 / 0.0173
    w.S = np.array([[-1, 1], [1, -1]], np.int32)
    _same(orc, w)
    w.S = np.array([[-1, 2], [1, -1]], np.int32)
    _same(orc, w)


def test_a_negative_count_is_the_oracle_s_error(orc):
    # an infection takes two susceptible animals of three
    w = W.plain_model(W.SISE, [[3, 0]], np.arange(30), W.sise_gdata(), seed=3,
                      v0=np.full((1, 1), 20.0))
    w.S = np.array([[-2, 0], [1, -1]], np.int32)
    code, _, _, _, err = orc.run(w)
    assert code == -4
    binding = _gpu()
    for tuning in (None, (1, 1), (16, 1 << 20)):
        with pytest.raises(binding.SimInfError) as e:
            binding.simulate(w, tuning=tuning)
        assert e.value.code == -4
        assert (e.value.err["node"], e.value.err["day"]) == (err["node"], err["day"])
