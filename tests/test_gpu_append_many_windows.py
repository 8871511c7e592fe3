"""A cache write whose windows hold more rows than its window-row CTAs take in one
pass: every row of every store, bit for bit."""
import pytest
import torch

from paper_2608_02691_gb300 import optr, synth

pytestmark = pytest.mark.gpu


def test_more_window_rows_than_one_pass():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2608_02691_gb300 import build
    build.build()
    sink, recent, B = 64, 256, 430
    n = sink + recent  # tokens per sequence: all of them are window rows, in order
    # 52 rows per CTA, at most 16 CTAs per SM
    assert B * n > 52 * 16 * torch.cuda.get_device_properties(0).multi_processor_count
    k, v = (x.cuda() for x in synth.kv_tokens(B * n, 1, "t4", 8, 0))
    R_k, R_v = synth.rotations(1, 8)
    p = optr.optr_params_create(R_k, R_v, synth.key_mean(k), 4, sink=sink, recent=recent)
    bt, pages = synth.page_tables([n] * B, True, 8)
    pool, win = optr.new_pool(p, pages), optr.new_windows(p, B)
    slot = torch.randperm(B, generator=torch.Generator().manual_seed(8)).int().cuda()
    optr.optr_kv_append_win(p, k, v, torch.arange(0, B * n + 1, n, dtype=torch.int32, device="cuda"),
                            torch.zeros(B, dtype=torch.int32, device="cuda"), bt.cuda(), pool, win, slot)
    torch.cuda.synchronize()
    assert optr.optr_device_error(p) == 0
    for kind, x in enumerate((k, v)):
        assert torch.equal(win[slot.long(), 0, kind], x.view(B, n, 128))
