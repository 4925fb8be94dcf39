"""The emulator network's calls hand raw pointers to the library: weights and
biases that it could not read (wrong device, type, layout or shape) raise
before the library is called.  Nothing runs on a GPU: the library is a stub
and the input only claims to be on one."""
import types

import pytest

torch = pytest.importorskip("torch")


class _Lib:
    """Accepts every call and counts them."""
    calls = 0

    def __getattr__(self, name):
        def call(*a):
            self.calls += name != "sg_mlp_gradients_scratch"
            return 0
        return call


def _claimed(t):
    """A stand-in for a CUDA tensor with t's type, layout and shape."""
    return types.SimpleNamespace(
        is_cuda=True, dtype=t.dtype, shape=t.shape, device="cpu", is_contiguous=t.is_contiguous,
        numel=t.numel, data_ptr=t.data_ptr)


@pytest.fixture
def net(monkeypatch):
    from paper_1605_01421_gb300 import binding, emulator
    stub = _Lib()
    monkeypatch.setattr(binding, "lib", lambda *a: stub)
    monkeypatch.setattr(emulator, "_s", lambda: None)
    emu = emulator.Emulator(device="cpu")
    emu.W8 = [torch.zeros(o, i, dtype=torch.uint8) for o, i in emulator.DIMS[1:]]
    emu.wscale = [torch.ones(o) for o, _ in emulator.DIMS[1:]]
    emu.act_scale = [1.0] * 3
    for name in ("W16", "b32", "W8", "wscale"):
        setattr(emu, name, [_claimed(t) for t in getattr(emu, name)])
    return emu, stub, _claimed(torch.zeros(8, 16, dtype=torch.bfloat16))


def _calls(emu, x):
    t = _claimed(torch.zeros(8, 3, dtype=torch.int32))
    return {"W16": (lambda: emu.forward(x), lambda: emu.gradients(x, t)),
            "b32": (lambda: emu.forward(x), lambda: emu.gradients(x, t),
                    lambda: emu.forward_fp8(x)),
            "W8": (lambda: emu.forward_fp8(x),), "wscale": (lambda: emu.forward_fp8(x),)}


def test_usable_weights_reach_the_library(net):
    emu, stub, x = net
    for calls in _calls(emu, x).values():
        for call in calls:
            before = stub.calls
            call()
            assert stub.calls == before + 1


@pytest.mark.parametrize("name,layer", [("W16", 0), ("W16", 2), ("b32", 0), ("b32", 3),
                                        ("W8", 1), ("wscale", 2)])
@pytest.mark.parametrize("fault", ["host", "type", "strided", "shape"])
def test_unusable_weights_raise(net, name, layer, fault):
    emu, stub, x = net
    good = getattr(emu, name)[layer]
    wide = torch.zeros([2 * n for n in good.shape], dtype=good.dtype)
    bad = {"host": lambda: torch.zeros(good.shape, dtype=good.dtype),
           "type": lambda: _claimed(torch.zeros(good.shape, dtype=torch.float64)),
           "strided": lambda: _claimed(wide[tuple(slice(None, None, 2) for _ in good.shape)]),
           "shape": lambda: _claimed(wide)}[fault]()
    getattr(emu, name)[layer] = bad
    for call in _calls(emu, x)[name]:
        with pytest.raises(ValueError):
            call()
    assert stub.calls == 0
    if name == "W16" and layer == 0:  # the E4M3 network's first layer
        with pytest.raises(ValueError):
            emu.forward_fp8(x)
