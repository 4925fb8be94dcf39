"""Tall contractions and the one-call gradients of the emulator network.

A contraction's FP32 result is within n 2^-23 sum |a b| of the exact one (n
additions, each rounded or cut to 24 bits; n is at most the number of
products plus the bias).  The one-call gradients use the same BF16
operands as the layer-by-layer calls, bit for bit, and differ from them in
the order of the FP32 sums only."""
import ctypes

import pytest

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


# one and several tiles of each width, ragged edges, K of whole stages, one
# element group more and less than the stages in flight
@pytest.mark.parametrize("M,N,K", [(1, 8, 1024), (128, 64, 1024), (129, 65, 1032), (392, 256, 8192),
                                   (256, 16, 8200), (256, 256, 1096), (3000, 100, 1024),
                                   (200, 72, 1016), (130, 130, 64), (130, 130, 200),
                                   (20000, 256, 256), (20000, 130, 72)])
def test_tall_contractions(gpu, M, N, K):
    import torch
    g = torch.Generator(device="cuda").manual_seed(M * 7 + N + K)
    A = torch.randn(M, K, generator=g, device="cuda").to(torch.bfloat16)
    B = torch.randn(N, K, generator=g, device="cuda").to(torch.bfloat16)
    bias = torch.randn(N, generator=g, device="cuda")
    C, _ = gpu.gemm_bf16(A, B, bias=bias)
    again, _ = gpu.gemm_bf16(A, B, bias=bias)
    assert torch.equal(C, again)
    a, b = A.double(), B.double()
    exact = a @ b.T + bias.double()
    bound = (K + 16) * 2.0 ** -23 * (a.abs() @ b.abs().T + bias.double().abs())
    assert bool(((C.double() - exact).abs() <= bound).all())


def _by_layers(gpu, em, emu, f, t):
    """The gradients call by call (transposes, contractions, column sums)."""
    import torch
    L = gpu.lib()
    B = f.shape[0]
    logits, acts, pres = emu.forward(f, keep=True)
    delta = torch.empty((B, em.NOUT), dtype=torch.bfloat16, device="cuda")
    loss = torch.zeros(1, dtype=torch.float64, device="cuda")
    em._check(L.sg_mlp_ce_loss(em._p(logits), em.NOUT, em._p(t), B, em._p(delta), em.NOUT,
                               em._p(loss), em._s()))
    deltas = [None] * 4
    for li in (3, 2, 1, 0):
        o, i = em.DIMS[li]
        deltas[li] = delta
        if li > 0:
            WT = emu.W16[li].t().contiguous()
            dpost, _ = gpu.gemm_bf16(delta, WT)
            nxt = torch.empty((B, i), dtype=torch.bfloat16, device="cuda")
            em._check(L.sg_gelu_backward(em._p(dpost), em._p(pres[li - 1]),
                                         ctypes.c_int64(B * i), em._p(nxt), em._s()))
            delta = nxt
    return float(loss.item()) / B, deltas, acts


@pytest.mark.parametrize("B", [8, 72, 128, 1024, 4104])
def test_one_call_gradients(gpu, B):
    import torch
    from paper_1605_01421_gb300 import emulator as em
    emu = em.Emulator("cuda", seed=B)
    g = torch.Generator(device="cuda").manual_seed(B)
    for b in emu.b32:
        b.copy_(0.05 * torch.randn(b.shape, generator=g, device="cuda"))
    f = torch.randn(B, em.NIN, generator=g, device="cuda").to(torch.bfloat16)
    t = torch.randint(0, em.BINS, (B, 3), generator=g, device="cuda", dtype=torch.int32)
    loss, dW, db = emu.gradients(f, t)
    loss2, deltas, acts = _by_layers(gpu, em, emu, f, t)
    assert abs(loss - loss2) <= 1e-12 * abs(loss2)
    for li in range(4):
        d, h = deltas[li].double(), acts[li].double()
        eps = (B + 16) * 2.0 ** -23
        assert bool(((dW[li].double() - d.T @ h).abs() <= eps * (d.abs().T @ h.abs())).all())
        assert bool(((db[li].double() - d.sum(0)).abs() <= eps * d.abs().sum(0)).all())


def test_refused_batches(gpu):
    import torch
    from paper_1605_01421_gb300 import emulator as em
    emu = em.Emulator("cuda", seed=1)
    f = torch.zeros(12, em.NIN, dtype=torch.bfloat16, device="cuda")
    t = torch.zeros(12, 3, dtype=torch.int32, device="cuda")
    with pytest.raises(gpu.SimInfError):
        emu.gradients(f, t)
