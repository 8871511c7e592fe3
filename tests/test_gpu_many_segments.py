"""Steps and decodes of more (sequence, KV head) segments than the GPU has SMs.

A query-rotation CTA then takes several sequences of a head, the last one fewer,
and the combine runs two CTAs per SM.  Every sequence's output has to be the one
that it gets in small batches of its own, where a CTA takes one sequence, up to
the split of its pages over the warps (both within the parity bound of the same
exact result, so within twice it of each other).
"""
import pytest
import torch

from paper_2608_02691_gb300 import optr, synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _setup():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2608_02691_gb300 import build
    build.build()
    torch.cuda.set_device(0)


@pytest.mark.parametrize("group,sink,recent", [(32, 0, 0), (128, 16, 48)])
@pytest.mark.parametrize("B,h_kv", [(77, 4), (113, 8), (128, 8)])
def test_large_batch_is_its_small_ones(group, sink, recent, B, h_kv):
    gen = torch.Generator().manual_seed(B + h_kv)
    lens = torch.randint(0, 900, (B,), generator=gen)
    lens[3] = 0
    total = int(lens.sum())
    k, v = synth.kv_tokens(total + B, h_kv, "t4", 7, 0)
    R_k, R_v = synth.rotations(h_kv, 7)
    p = optr.optr_params_create(R_k, R_v, synth.key_mean(k), 4 * h_kv, group=group, sink=sink,
                                recent=recent)
    bt, pages = synth.page_tables([int(n) + 1 for n in lens], True, 7)
    k, v, bt = k.cuda(), v.cuda(), bt.cuda()
    i32 = dict(dtype=torch.int32, device="cuda")
    cu = torch.cat([torch.zeros(1, dtype=torch.long), lens.cumsum(0)]).to(**i32)
    q = torch.randn(B, 4 * h_kv, 128, generator=gen).bfloat16().cuda()
    win = slots = None
    pool = optr.new_pool(p, pages)
    ctx = (p, k[:total], v[:total], cu, torch.zeros(B, **i32), bt, pool)
    if sink + recent:
        win, slots = optr.new_windows(p, B), torch.arange(B, **i32)
        optr.optr_kv_append_win(*ctx, win, slots)
    else:
        optr.optr_kv_append(*ctx)

    def step(lo, hi, pool, win):
        n = hi - lo
        out = torch.empty(n, 4 * h_kv, 128, device="cuda")
        a = (p, q[lo:hi], k[total + lo:total + hi], v[total + lo:total + hi],
             torch.arange(n + 1, **i32), lens[lo:hi].to(**i32), bt[lo:hi].contiguous(),
             (lens[lo:hi] + 1).to(**i32), pool)
        ws = optr.new_workspace(p, n, bt.shape[1])
        if win is not None:
            optr.optr_decode_step_win(*a, win, slots[lo:hi].contiguous(), out, ws)
        else:
            optr.optr_decode_step(*a, out, ws)
        return out

    pool2, win2 = pool.clone(), None if win is None else win.clone()
    big = step(0, B, pool, win)
    small = torch.cat([step(b, min(b + 4, B), pool2, win2) for b in range(0, B, 4)])
    torch.cuda.synchronize()
    assert optr.optr_device_error(p) == 0
    assert torch.equal(pool, pool2)
    if win is not None:
        assert torch.equal(win, win2)
    # the parity bound: 2e-3 of the output's RMS at any element, per side
    assert (big - small).abs().max() <= 4e-3 * small.pow(2).mean().sqrt()
