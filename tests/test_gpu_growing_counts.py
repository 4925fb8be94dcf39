"""Models from transition strings whose counts leave the range that FP32 holds
exactly within one day: counts stay int32 on every path, as in the oracle."""
import numpy as np
import pytest

from paper_1605_01421_gb300 import workloads as W

pytestmark = pytest.mark.gpu

# odd steps across 2^24 = 16,777,216 and, there, single steps in both
# directions whose rates read the count; counts are not conserved
_UP = ["@ -> a -> 127*X", "@ -> b -> X", "X -> d*X -> @"]


@pytest.mark.parametrize("tuning", [None, (64, 1 << 20), (16, 1)])
@pytest.mark.parametrize("start", [(1 << 23) - 1, (1 << 23) - 40000, (1 << 24) - 3001, 1 << 25])
def test_counts_beyond_2_to_the_24(orc, tuning, start):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1605_01421_gb300 import binding
    # below 2^23 at the start: 75,000 steps of 127 end near 18 million
    a = 75000.0 if start < 1 << 23 else 40.0
    g = {"a": a, "b": 900.0, "d": 5e-5}
    u0 = np.array([[start - i] for i in range(3)])
    w = W.parsed_model(_UP, ["X"], g, u0, np.arange(0, 2), seed=17)
    code, U0, _, R0, err = orc.run(w)
    assert code == 0, err
    assert U0[0, -1].min() > 1 << 24 or start > 1 << 24 or a < 100.0
    U1, _, st = binding.simulate(w, tuning=tuning)
    assert np.array_equal(U0, U1)
    assert st["reactions"] == int(R0.sum())
