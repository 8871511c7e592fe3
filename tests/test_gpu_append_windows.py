"""Long cache writes that find the window rows from the windows, in the same
launch (calls that write at least as many tokens as their windows hold), at the
edges: exactly as many tokens, one fewer (the separate copy), sink only, recent
only, one and an odd number of KV heads, writes that begin inside and past the
sink and end inside the recent window, sequences without new tokens, and a bad
slot.  The store is a copy, so every bit is compared with the oracle's.
"""
import numpy as np
import pytest
import torch

from oracle import oracle
from paper_2608_02691_gb300 import optr, synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _setup():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2608_02691_gb300 import build
    build.build()
    torch.cuda.set_device(0)


@pytest.mark.parametrize("h_kv,sink,recent,lens,pos0", [
    (8, 16, 240, [512], [0]),              # B * rows = 256 of 512 tokens
    (1, 64, 256, [320, 320], [0, 64]),     # exactly as many
    (1, 64, 256, [319, 320], [0, 64]),     # one fewer: the separate copy
    (3, 32, 0, [300, 0, 5], [0, 9, 30]),
    (5, 0, 48, [129, 700], [1000, 3]),
    (2, 64, 256, [900, 1, 0, 2000], [40, 5000, 7, 63]),
])
@pytest.mark.parametrize("bad_slot", [False, True])
def test_window_rows_of_long_writes(h_kv, sink, recent, lens, pos0, bad_slot):
    B = len(lens)
    k, v = synth.kv_tokens(sum(lens), h_kv, "t4", 6, 0)
    cu = np.concatenate([[0], np.cumsum(lens)]).astype(np.int32)
    p0 = np.array(pos0, np.int32)
    slots = np.arange(B, dtype=np.int32)[::-1].copy()
    ref = oracle.new_windows(B, h_kv, sink, recent)
    oracle.window_write(synth.bf16_bits(k), synth.bf16_bits(v), cu, p0, ref, slots, sink, recent)
    R_k, R_v = synth.rotations(h_kv, 6)
    p = optr.optr_params_create(R_k, R_v, synth.key_mean(k), 4 * h_kv, sink=sink, recent=recent)
    bt, num_pages = synth.page_tables([a + b for a, b in zip(pos0, lens)], True, 6)
    pool = optr.new_pool(p, num_pages)
    win = optr.new_windows(p, B)
    given = slots.copy()
    if bad_slot:
        ref[slots[0]] = 0
        given[0] = B
    optr.optr_kv_append_win(p, k.cuda(), v.cuda(), torch.from_numpy(cu).cuda(),
                            torch.from_numpy(p0).cuda(), bt.cuda(), pool, win,
                            torch.from_numpy(given).cuda())
    torch.cuda.synchronize()
    assert (optr.optr_device_error(p) != 0) == bad_slot
    np.testing.assert_array_equal(win.cpu().view(torch.int16).numpy().view(np.uint16), ref)
