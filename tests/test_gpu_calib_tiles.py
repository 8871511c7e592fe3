"""The calibration's products in 64 x 32 tiles, at row, column and depth counts that
are no multiple of a tile or a 128-deep chunk, several heads at once, with the
subtraction and the mask of the epilogue: loss and generator gradient against the
float64 oracle, 1e-9 of the largest magnitude (tests/test_gpu_calibration.py states
why).  Smaller calls take 32 x 16 tiles, which every other calibration test runs.
"""
import pytest
import torch

from oracle import calibration as cal
from paper_2608_02691_gb300 import optr, synth

pytestmark = pytest.mark.gpu

F64 = torch.float64
D = 128
REL = 1e-9


@pytest.fixture(scope="module", autouse=True)
def _setup():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2608_02691_gb300 import build
    build.build()
    torch.cuda.set_device(0)


def _products(T, nt, g, dm):
    """(rows, columns, depth, batch) of the products of one evaluation."""
    return [(T, D, D, 1), (nt, T, D, g), (nt, D, T, g), (nt, dm, D, g), (nt, D, dm, g),
            (T, D, g * nt, 1), (D, D, 2 * T, 1)]


@pytest.mark.parametrize("which", [0, 1])
@pytest.mark.parametrize("group,clip,sink,recent", [(32, 1.0, 0, 0), (128, 0.95, 7, 90)])
@pytest.mark.parametrize("T,nt,g,dm", [(1281, 65, 4, 1001), (1250, 127, 3, 433)])
def test_large_tiles_with_remainders(which, group, clip, sink, recent, T, nt, g, dm):
    for m, n, k, b in _products(T, nt, g, dm):  # 64 x 32 tiles x chunks fill half the SMs
        assert -(-m // 64) * -(-n // 32) * b * -(-k // 128) >= 76, (m, n, k, b)
    q, K, V, W_O, t_pos = synth.calib_trace(13, T=T, nt=nt, g=g, d_model=dm)
    mu = K.mean(0)
    gen = torch.Generator().manual_seed(14)
    R0 = cal.hadamard(D)
    A = torch.randn(D, D, generator=gen, dtype=F64) * 0.05
    R_K = cal.rotation(R0, torch.randn(D, D, generator=gen, dtype=F64) * 0.05)
    Ar = A.clone().requires_grad_(True)
    R = cal.rotation(R0, Ar)
    if which == 0:
        L = cal.key_loss(q, K, V, mu, R, W_O, t_pos.long(), 0.7, clip, group, sink, recent)
    else:
        L = cal.value_loss(q, K, V, mu, R_K, R, W_O, t_pos.long(), clip, clip, group, sink, recent)
    (ref,) = torch.autograd.grad(L, Ar)
    cfg = optr.calib_config(g, dm, T, nt, group=group, sink=sink, recent=recent, lam=0.7, clip_k=clip,
                            clip_v=clip)
    loss, dA = optr.optr_calib_loss_grad(cfg, which, *[x.cuda() for x in (q, K, V, t_pos, W_O, mu, R0, A)],
                                         R_K=R_K.cuda())
    lr = float(L.detach())
    assert abs(float(loss.item()) - lr) <= REL * abs(lr)
    assert float((dA.cpu() - ref).abs().max()) <= REL * float(ref.abs().max())
