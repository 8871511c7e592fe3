"""The one-launch decode of small batches against the oracle: every cluster
size (8, 4, 2 and 1 CTAs per sequence and KV head), lengths around page, warp
and chunk boundaries (none, one token, a page and its neighbours, more than 32
pages for a warp's page table), both record sizes, BF16 windows that cover
nothing, some or all of a sequence.  Tolerance as for every decode
(parity_helpers): max |error| <= 2e-3 of the oracle's RMS."""
import numpy as np
import pytest
import torch

import parity_helpers as ph
from oracle import oracle
from paper_2608_02691_gb300 import optr, synth

pytestmark = pytest.mark.gpu

BATCHES = {
    "8 CTAs": [2081],
    "8 CTAs, one page": [16],
    "4 CTAs": [1, 0, 1025],
    "2 CTAs": [17, 300, 15, 16, 1, 640],
    "1 CTA": [33, 0, 129, 513, 16, 1, 47, 255, 256, 257, 31, 32],
}


@pytest.fixture(scope="module", autouse=True)
def _setup():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2608_02691_gb300 import build
    build.build()
    oracle.build()
    torch.cuda.set_device(0)


@pytest.mark.parametrize("name", BATCHES)
@pytest.mark.parametrize("group,sink,recent", [(32, 0, 0), (128, 0, 0), (32, 16, 100), (128, 64, 256)])
def test_one_launch_decode(name, group, sink, recent):
    ctx = BATCHES[name]
    c = synth.build_case(synth.Workload(name, len(ctx), ctx, "t4", shuffle=True), 3)
    pool_ref, _, _ = ph.oracle_case(c, group=group)
    n_slots = c["B"] + 1
    slots = np.arange(n_slots, dtype=np.int32)[::-1][:c["B"]].copy()
    win = None
    if sink + recent:
        win = oracle.new_windows(n_slots, c["h_kv"], sink, recent)
        oracle.window_write(synth.bf16_bits(c["k_ctx"]), synth.bf16_bits(c["v_ctx"]),
                            c["cu_ctx"].numpy(), c["pos0_ctx"].numpy(), win, slots, sink, recent)
    ref = oracle.decode_attention(
        synth.bf16_bits(c["q"]), c["block_table"].numpy(), c["seq_lens"].numpy(), pool_ref,
        c["R_k"].numpy(), c["R_v"].numpy(), c["h_kv"],
        **(dict(win=win, win_slot=slots, sink=sink, recent=recent, mu=c["mu"].numpy())
           if win is not None else {}))
    dev = "cuda"
    p = optr.optr_params_create(c["R_k"], c["R_v"], c["mu"], c["h_q"], sink=sink, recent=recent,
                                group=group)
    bt, lens = c["block_table"].to(dev), c["seq_lens"].to(dev)
    out = torch.full((c["B"], c["h_q"], 128), 7.0, dtype=torch.float32, device=dev)
    ws = optr.new_workspace(p, c["B"], bt.shape[1])
    pool = torch.from_numpy(pool_ref).to(dev)
    if win is None:
        optr.optr_decode_attention(p, c["q"].to(dev), bt, lens, pool, out, ws)
    else:
        w = torch.from_numpy(win.view(np.int16)).view(torch.bfloat16).to(dev)
        optr.optr_decode_attention_win(p, c["q"].to(dev), bt, lens, pool, w,
                                       torch.from_numpy(slots).to(dev), out, ws)
    torch.cuda.synchronize()
    assert optr.optr_device_error(p) == 0
    got = out.cpu().double().numpy()
    for b, n in enumerate(ctx):
        if n == 0:
            assert not got[b].any()
    ph.assert_decode_close(got, ref, name)
