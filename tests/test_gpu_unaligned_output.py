"""A trajectory buffer U that is not 8-byte aligned takes the sparse schedule's
scan with a unit per lane instead of the paired one; the results are the
same."""
import numpy as np
import pytest

from paper_1605_01421_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind,tuning", [(W.SIS, (130, 4)), (W.SISE, (400, 4)),
                                         (W.SISE3, (400, 4)), (W.SISE3, (257, 2))])
def test_unaligned_trajectory(orc, kind, tuning):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1605_01421_gb300 import binding
    rng = np.random.default_rng(kind)
    n, C = 200, 6 if kind == W.SISE3 else 2
    u0 = rng.integers(0, 60, (n, C))
    u0[::3, 1::2] = 0  # herds without infected animals
    g = {W.SIS: [0.003, 0.3], W.SISE: W.sise_gdata(), W.SISE3: W.sise3_gdata()}[kind]
    w = W.plain_model(kind, u0, np.arange(0, 8), g, seed=9, n_rep=4)
    code, U0, V0, R0, err = orc.run(w)
    assert code == 0, err
    m = binding.Model(w)
    m.set_tuning(*tuning)
    dev = lambda a, t: torch.as_tensor(np.ascontiguousarray(a, t), device="cuda")  # noqa: E731
    room = torch.empty(U0.size + 1, dtype=torch.int32, device="cuda")
    U = room[1:].view(U0.shape)
    assert U.data_ptr() % 8 == 4
    V = torch.empty(V0.shape, dtype=torch.float64, device="cuda")
    rc, st, er = m.run(w.tspan, w.seed, 4, dev(w.u0, np.int32), dev(w.v0, np.float64), U, V)
    m.close()
    assert np.array_equal(U.cpu().numpy(), U0)
    assert np.array_equal(V.cpu().numpy().view(np.uint64), V0.view(np.uint64))
