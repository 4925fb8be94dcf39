"""The direct method's decisions from FP32 intervals (sg_filter.cuh): the
enclosures hold on the device (logarithm, reciprocal), and the trajectories
are the oracle's bit for bit where the intervals apply, where they do not
(large counts, a caller's own S and G, negative zero phi, very late times,
days of very many draws) and where a warp with exact times takes over."""
import numpy as np
import pytest

from paper_1605_01421_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gpu():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1605_01421_gb300 import binding
    binding.build()
    binding.lib()
    return binding


def _same(orc, gpu, w, tuning=None):
    code, U0, V0, R0, err0 = orc.run(w)
    assert code == 0, err0
    U1, V1, st = gpu.simulate(w, tuning=tuning)
    assert np.array_equal(U0, U1)
    assert np.array_equal(V0.view(np.uint64), V1.view(np.uint64))
    assert st["reactions"] == int(R0.sum())


def _neglog(words):
    k = (words[:, 1].astype(np.uint64) << np.uint64(20)) | (words[:, 0].astype(np.uint64)
                                                           >> np.uint64(12))
    m = 2 * k + np.uint64(1)  # r1 = m 2^-53
    far = np.uint64(1 << 53) - m
    near = -np.log1p(-far.astype(np.float64) * 2.0 ** -53)
    return np.where(m > np.uint64(1 << 52), near, -np.log(m.astype(np.float64) * 2.0 ** -53))


def test_enclosures_hold_on_the_device(gpu):
    # every FP32 argument of the logarithm in [1/2, 1) and 2^16 of each
    # binary order below; every FP32 mantissa of the reciprocal, over the
    # orders it is used in; the low words random
    rng = np.random.default_rng(1)
    hi = [np.arange(1 << 31, 1 << 32, 1 << 8, dtype=np.uint64)]
    for e in range(0, 31):
        n = min(1 << e, 1 << 16)
        hi.append((1 << e) + np.linspace(0, (1 << e) - 1, n).astype(np.uint64))
    hi = np.concatenate(hi + [np.zeros(1 << 16, np.uint64), np.array([2 ** 32 - 1], np.uint64)])
    words = np.stack([rng.integers(0, 1 << 32, hi.size, dtype=np.uint64), hi], 1)
    words[-1, 0] = 2 ** 32 - 1
    words[-2, 0] = 0
    n = hi.size
    mant = (np.arange(n, dtype=np.uint32) & np.uint32((1 << 23) - 1)) | np.uint32(127 << 23)
    x = np.ldexp(mant.view(np.float32), rng.integers(-100, 100, n).astype(np.int32))
    b = gpu.filter_bounds_batch(words, x).astype(np.float64)
    E = _neglog(words)
    assert np.all(b[:, 0] <= E) and np.all(E <= b[:, 1])
    # the stated widths: 2 (3.2e-7 + 2^-21 E), 4 ulps of the reciprocal
    assert np.all(b[:, 1] - b[:, 0] <= 1e-6 + 2e-6 * E)
    one = 1.0 / x.astype(np.float64)
    assert np.all(b[:, 2] <= one) and np.all(one <= b[:, 3])
    assert np.all(b[:, 3] - b[:, 2] <= 2.0 ** -20 * one)


def _u0(rng, n, C, herd):
    return rng.integers(0, herd, (n, C)).astype(np.int32)


@pytest.mark.parametrize("kind", [W.SIR, W.SIS, W.SISE, W.SISE3])
@pytest.mark.parametrize("tuning", [None, (16, 3), (129, 3), (700, 1)])
def test_kinds_with_and_without_hand_over(orc, gpu, kind, tuning):
    # heavy_after 1 and 3 hand most active days to warps with exact times,
    # more of them than the sparse schedule has slots
    rng = np.random.default_rng(10 + kind)
    C = {W.SIR: 3, W.SISE3: 6}.get(kind, 2)
    g = {W.SIR: [0.4, 0.2], W.SIS: [0.002, 0.3],
         W.SISE: W.sise_gdata(), W.SISE3: W.sise3_gdata()}[kind]
    nv = 1 if kind in (W.SISE, W.SISE3) else 0
    w = W.plain_model(kind, _u0(rng, 701, C, 200), np.arange(3, 15), g, seed=99, n_rep=2,
                      v0=rng.uniform(0, 3, (701, nv)))
    _same(orc, gpu, w, tuning)


@pytest.mark.parametrize("herd,t0,days", [(1 << 21, 0, 1), (60000, 5, 2), (3, 2 ** 30, 6),
                                          (40, 2 ** 31 - 99, 8), (40, -7, 12)])
def test_ranges_where_intervals_widen_or_end(orc, gpu, herd, t0, days):
    # counts beyond the FP32 form, days of more draws than the thread takes,
    # unit times where FP64's own rounding of t is 2^-22, negative times
    rng = np.random.default_rng(herd)
    n = 6 if herd > 1000 else 500
    u0 = np.stack([np.full(n, herd), rng.integers(1, 5, n) * max(1, herd // 4)], 1)
    gam = 1e-4 if herd > 1 << 20 else 0.9
    w = W.plain_model(W.SISE, u0, t0 + np.arange(days + 1), W.sise_gdata(gamma=gam), seed=3,
                      v0=np.full((n, 1), 0.01))
    _same(orc, gpu, w)


@pytest.mark.parametrize("tuning", [None, (200, 2)])
def test_own_tables_and_negative_zero_phi(orc, gpu, tuning):
    rng = np.random.default_rng(5)
    u0 = _u0(rng, 600, 2, 60)
    w = W.plain_model(W.SISE, u0, np.arange(8), W.sise_gdata(), seed=4,
                      v0=np.where(rng.random((600, 1)) < 0.5, -0.0, 0.7))
    _same(orc, gpu, w, tuning)
    # G leaves rate 0 as it was after transition 1: rates depend on the path
    w.G = np.array([[1, 0], [1, 1]], np.int32)
    _same(orc, gpu, w, tuning)
    # a recovery that removes the animal
    w.G = np.ones((2, 2), np.int32)
    w.S = np.array([[-1, 0], [1, -1]], np.int32)
    _same(orc, gpu, w, tuning)


@pytest.mark.parametrize("trans,comps,g,u0", [
    # differences and quotients in the propensity, negative intermediate
    # values, a constant that is no FP32 number, growth and extinction
    (["@ -> a*(2-b) -> X", "X -> 0.1*X*(X-1)/(X+1) -> @", "X -> -(c-d)*X -> Y",
      "Y -> Y/(1+X*X/K) -> @"], ["X", "Y"],
     {"a": 40.3, "b": 0.7, "c": 0.2, "d": 0.9, "K": 50.0}, (3, 0)),
    (W.MPARSE_PREDATOR_PREY, ["R", "F"], W.PREDATOR_PREY_GDATA, (900, 90)),
    (["S -> b*S*I/(S+I) -> I", "I -> g*I -> S"], ["S", "I"], {"b": 0.6, "g": 0.2},
     (3000, 20)),
])
def test_parsed_models(orc, gpu, trans, comps, g, u0):
    rng = np.random.default_rng(8)
    u = np.array(u0) + rng.integers(0, 5, (60, len(comps)))
    w = W.parsed_model(trans, comps, g, u, np.arange(0, 6), seed=21)
    _same(orc, gpu, w)
