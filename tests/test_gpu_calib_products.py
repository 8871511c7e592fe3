"""The calibration's float64 products (split into fp16 digits, 128-deep chunks;
at these sizes nearly all in 32 x 16 tiles, test_gpu_calib_tiles.py has the 64 x 32
ones) where they can go wrong: rows, columns and depths that are no multiple of a
tile or a chunk, one row or one token, more output channels than one chunk, split
depths, operands whose magnitudes differ as wholes (test_gpu_calib_exact.py has the
ones that differ inside a row), and non-finite input.  Loss and generator gradient against the float64 oracle; both sides
round differently at a few 1e-16 per product, and 1e-9 of the largest
magnitude is allowed (tests/test_gpu_calibration.py states why).
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


def _run(which, T, nt, g, d_model, ks=1.0, vs=1.0, ws=1.0, bad=None):
    q, K, V, W_O, t_pos = synth.calib_trace(3, T=T, nt=nt, g=g, d_model=d_model)
    K, q, V, W_O = K * ks, q / ks, V * vs, W_O * ws
    if bad is not None:
        V[T // 2, 5] = bad
    mu = K.mean(0)
    gen = torch.Generator().manual_seed(4)
    R0 = cal.hadamard(D)
    A = torch.randn(D, D, generator=gen, dtype=F64) * 0.05
    R_K = cal.rotation(R0, torch.randn(D, D, generator=gen, dtype=F64) * 0.05)
    cfg = optr.calib_config(g, d_model, T, nt, lam=0.7)
    dev = [x.cuda() for x in (q, K, V, t_pos, W_O, mu, R0, A)]
    loss, dA = optr.optr_calib_loss_grad(cfg, which, *dev, R_K=R_K.cuda())
    Ar = A.clone().requires_grad_(True)
    R = cal.rotation(R0, Ar)
    if which == 0:
        L = cal.key_loss(q, K, V, mu, R, W_O, t_pos.long(), 0.7, 1.0, 32, 0, 0)
    else:
        L = cal.value_loss(q, K, V, mu, R_K, R, W_O, t_pos.long(), 1.0, 1.0, 32, 0, 0)
    return float(loss.item()), dA.cpu(), L, Ar


@pytest.mark.parametrize("which", [0, 1])
@pytest.mark.parametrize("T,nt,g,d_model,ks,vs,ws", [
    (40, 1, 1, 1, 1.0, 1.0, 1.0),
    (33, 33, 1, 31, 1.0, 1.0, 1.0),
    (63, 17, 3, 65, 1.0, 1.0, 1.0),
    (64, 32, 2, 128, 1.0, 1.0, 1.0),
    (65, 16, 4, 127, 1.0, 1.0, 1.0),
    (1025, 9, 2, 1000, 1.0, 1.0, 1.0),
    (200, 31, 4, 300, 1.0, 1e3, 1e-30),
    (200, 31, 4, 300, 1.0, 1e-2, 1e40),
])
def test_products_at_tile_edges(which, T, nt, g, d_model, ks, vs, ws):
    loss, dA, L, Ar = _run(which, T, nt, g, d_model, ks, vs, ws)
    # torch's derivative of matrix_exp scales the block matrix of generator and
    # incoming gradient by the norm of both, so a gradient of 1e72 costs it 240
    # squarings (3e-8 of error): it gets the gradient of L / L instead
    lr = float(L.detach())
    (ref,) = torch.autograd.grad(L / lr, Ar)
    ref = ref * lr
    assert abs(loss - lr) <= REL * abs(lr)
    assert float((dA - ref).abs().max()) <= REL * float(ref.abs().max())


@pytest.mark.parametrize("which", [0, 1])
@pytest.mark.parametrize("bad", [float("nan"), float("inf")])
def test_non_finite_input_does_not_give_a_finite_loss(which, bad):
    loss, _, _, _ = _run(which, 100, 20, 2, 40, bad=bad)
    assert loss != loss or abs(loss) == float("inf")


@pytest.mark.parametrize("T,nt,d_model,steps,group", [
    (97, 16, 160, 5, 32),    # W^T W replaces W; odd token count
    (97, 16, 128, 5, 128),
    (130, 9, 127, 6, 32),    # too few output channels for it
    (64, 4, 300, 4, 128),    # too few query rows for it
])
def test_calibration_with_and_without_output_products(T, nt, d_model, steps, group):
    q, K, V, W_O, t_pos = synth.calib_trace(8, T=T, nt=nt, g=2, d_model=d_model)
    ref = cal.calibrate_head(q, K, V, W_O, t_pos.long(), steps=steps, lr=0.01, group=group,
                             select_every=2)
    cfg = optr.calib_config(2, d_model, T, nt, steps=steps, select_every=2, group=group, lr=0.01)
    got = optr.optr_calibrate_head(cfg, *[x.cuda() for x in (q, K, V, t_pos, W_O)])
    R_K, R_V, mu, hk, hv = [torch.as_tensor(x, dtype=F64) for x in ref]
    gR_K, gR_V, gmu, ghk, ghv = [x.cpu() for x in got]
    assert float((gmu - mu).abs().max()) <= 1e-12 * float(mu.abs().max())
    assert float(((ghk - hk) / hk).abs().max()) <= REL
    assert float(((ghv - hv) / hv).abs().max()) <= REL
    assert float((gR_K - R_K).abs().max()) <= REL
    assert float((gR_V - R_V).abs().max()) <= REL
