"""The decode that splits a batch's pages over all SMs (query rotation, partials,
combine: three launches), at lengths that the oracle finishes quickly.

Small batches with short block tables are one launch instead; the width of the
table decides, not the lengths, and a table of more than 1440 pages is always
split, whether its sequences have the pages or not.  A batch of few segments then has
its combine spread over several CTAs per (sequence, KV head): with both record
sizes, BF16 windows and the folded value rotation.  Tolerance as for every decode
(parity_helpers): max |error| <= 2e-3 of the oracle's RMS.
"""
import numpy as np
import pytest
import torch

import parity_helpers as ph
from oracle import oracle
from paper_2608_02691_gb300 import optr, synth

pytestmark = pytest.mark.gpu

WIDE = 1500


@pytest.fixture(scope="module", autouse=True)
def _setup():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2608_02691_gb300 import build
    build.build()
    oracle.build()
    oracle.set_threads(max(1, min(16, __import__("os").cpu_count() or 1)))
    torch.cuda.set_device(0)


def _wide(bt):
    out = torch.full((bt.shape[0], WIDE), -1, dtype=torch.int32)
    out[:, :bt.shape[1]] = bt
    return out.cuda()


@pytest.mark.parametrize("fold", [False, True])
@pytest.mark.parametrize("group,sink,recent", [
    (32, 0, 0), (128, 0, 0), (32, 64, 256), (128, 64, 256), (128, 16, 100)])
@pytest.mark.parametrize("lens", [[4113], [2081, 0, 300, 16], [0]])
def test_combine_over_several_ctas(lens, group, sink, recent, fold):
    c = synth.build_case(synth.Workload("split", len(lens), lens, "t4", shuffle=True), 5)
    ref_c = dict(c)
    if fold:
        ref_c["R_v"] = torch.eye(128).expand(c["h_kv"], 128, 128).contiguous()
    pool_ref, _, _ = ph.oracle_case(ref_c, group=group)
    win = slots = None
    if sink + recent:
        slots = np.arange(len(lens), dtype=np.int32)[::-1].copy()
        win = oracle.new_windows(len(lens), c["h_kv"], sink, recent)
        if sum(lens):
            oracle.window_write(synth.bf16_bits(c["k_ctx"]), synth.bf16_bits(c["v_ctx"]),
                                c["cu_ctx"].numpy(), c["pos0_ctx"].numpy(), win, slots, sink, recent)
    ref = oracle.decode_attention(
        synth.bf16_bits(c["q"]), c["block_table"].numpy(), c["seq_lens"].numpy(), pool_ref,
        c["R_k"].numpy(), ref_c["R_v"].numpy(), c["h_kv"],
        **(dict(win=win, win_slot=slots, sink=sink, recent=recent, mu=c["mu"].numpy())
           if win is not None else {}))
    p = optr.optr_params_create(c["R_k"], None if fold else c["R_v"], c["mu"], c["h_q"], group=group,
                                sink=sink, recent=recent)
    bt = _wide(c["block_table"])
    out = torch.full((c["B"], c["h_q"], 128), 7.0, device="cuda")
    args = [c["q"].cuda(), bt, c["seq_lens"].cuda(), torch.from_numpy(pool_ref).cuda()]
    ws = optr.new_workspace(p, c["B"], WIDE).fill_(0xFF)
    if win is None:
        optr.optr_decode_attention(p, *args, out, ws)
    else:
        optr.optr_decode_attention_win(
            p, *args, torch.from_numpy(win.view(np.int16)).view(torch.bfloat16).cuda(),
            torch.from_numpy(slots).cuda(), out, ws)
    torch.cuda.synchronize()
    assert optr.optr_device_error(p) == 0
    got = out.cpu().double().numpy()
    for b, n in enumerate(lens):
        if n == 0:
            assert not got[b].any()
    if sum(lens):
        ph.assert_decode_close(got, ref, f"{lens} G {group} windows {sink}, {recent}")


CONFIGS = [dict(), dict(group=128, clip_k=0.96, clip_v=0.92), dict(sink=64, recent=256),
           dict(group=128, sink=16, recent=100, clip_k=0.96, clip_v=0.92), dict(fold=True)]


def _filled(B, h_kv, lens, new, cfg, seed):
    """Params, the step's arguments (new tokens per sequence after lens[b]) and the
    written context's pool and window store."""
    cfg = dict(cfg)
    fold = cfg.pop("fold", False)
    total = sum(lens)
    k, v = synth.kv_tokens(total + B * new, h_kv, "t4", seed, 0)
    R_k, R_v = synth.rotations(h_kv, seed)
    p = optr.optr_params_create(R_k, None if fold else R_v, synth.key_mean(k), 4 * h_kv, **cfg)
    bt, pages = synth.page_tables([n + new for n in lens], True, seed)
    i32 = lambda x: torch.as_tensor(x, dtype=torch.int32, device="cuda")
    pool, win, slot = optr.new_pool(p, pages), None, None
    ctx = (p, k[:total].cuda(), v[:total].cuda(), i32(np.concatenate([[0], np.cumsum(lens)])),
           i32([0] * B), bt.cuda(), pool)
    if p.cfg.sink + p.cfg.recent:
        win, slot = optr.new_windows(p, B), i32(np.arange(B)[::-1].copy())
        optr.optr_kv_append_win(*ctx, win, slot)
    else:
        optr.optr_kv_append(*ctx)
    step = dict(q=synth.queries(B, 4 * h_kv, seed).cuda(), k=k[total:].cuda(), v=v[total:].cuda(),
                cu=i32(np.arange(B + 1) * new), pos0=i32(lens), seq=i32([n + new for n in lens]))
    return p, step, bt, pool, win, slot


def _step(p, s, bt, pool, win, slot, out, ws):
    a = (p, s["q"], s["k"], s["v"], s["cu"], s["pos0"], bt, s["seq"], pool)
    if win is not None:
        optr.optr_decode_step_win(*a, win, slot, out, ws)
    else:
        optr.optr_decode_step(*a, out, ws)


@pytest.mark.parametrize("cfg", CONFIGS, ids=lambda c: "-".join(f"{k}{v}" for k, v in c.items()) or "plain")
@pytest.mark.parametrize("B,host", [(16, False), (16, True), (21, False)])
def test_step_replays_from_a_cuda_graph(B, host, cfg):
    """Cache write, partials and combine of a step captured once and replayed:
    bytes and output of direct calls, with up to one and more than one segment
    per SM, with device and pinned host activations."""
    lens = [257 + 31 * b for b in range(B)]
    p, s, bt, pool, win, slot = _filled(B, 8, lens, 1, cfg, 3)
    bt = _wide(bt)
    ws = optr.new_workspace(p, B, WIDE)
    out = torch.empty(B, 32, 128, device="cuda")
    pool_g, win_g = pool.clone(), None if win is None else win.clone()
    for _ in range(2):
        _step(p, s, bt, pool, win, slot, out, ws)
    out_g = torch.zeros(B, 32, 128)
    out_g = out_g.pin_memory() if host else out_g.cuda()
    if host:
        s = {n: x.cpu().pin_memory() if n in ("q", "k", "v") else x for n, x in s.items()}
    torch.cuda.synchronize()
    st, g = torch.cuda.Stream(), torch.cuda.CUDAGraph()
    with torch.cuda.stream(st):
        _step(p, s, bt, pool_g, win_g, slot, out_g, ws)  # outside the capture
        st.synchronize()
        with torch.cuda.graph(g, stream=st):
            _step(p, s, bt, pool_g, win_g, slot, out_g, ws)
    for _ in range(2):
        out_g.zero_()
        torch.cuda.synchronize()
        g.replay()
        torch.cuda.synchronize()
        assert torch.equal(out.cpu(), out_g.cpu())
    assert optr.optr_device_error(p) == 0
    assert torch.equal(pool, pool_g)
    assert win is None or torch.equal(win, win_g)


@pytest.mark.parametrize("cfg", CONFIGS, ids=lambda c: "-".join(f"{k}{v}" for k, v in c.items()) or "plain")
@pytest.mark.parametrize("B,new", [
    (16, 12), (16, 4), (5, 13),  # 192, 64 and 65 new tokens: cache-write tiles of 16, 4 and 16
    (2, 128), (1, 256),          # the largest step in one launch, over 8 and 16 pages
    (21, 3), (21, 12),           # more segments than SMs
])
@pytest.mark.parametrize("wide", [False, True])
def test_step_of_several_tokens_is_write_then_decode(B, new, cfg, wide):
    """A step that writes several tokens per sequence across page boundaries
    equals the cache write followed by the decode bit for bit: pages that the
    step writes are read only after it."""
    lens = [16 * (b % 5) * 7 + 15 for b in range(B)]  # the write starts on a page's last slot
    p, s, bt, pool, win, slot = _filled(B, 8, lens, new, cfg, 4)
    bt = _wide(bt) if wide else bt.cuda()
    ws = optr.new_workspace(p, B, bt.shape[1])
    pool2, win2 = pool.clone(), None if win is None else win.clone()
    out, out2 = torch.empty(B, 32, 128, device="cuda"), torch.full((B, 32, 128), 7.0, device="cuda")
    w = (p, s["k"], s["v"], s["cu"], s["pos0"], bt, pool)
    d = (p, s["q"], bt, s["seq"], pool)
    if win is not None:
        optr.optr_kv_append_win(*w, win, slot)
        optr.optr_decode_attention_win(*d, win, slot, out, ws)
    else:
        optr.optr_kv_append(*w)
        optr.optr_decode_attention(*d, out, ws)
    _step(p, s, bt, pool2, win2, slot, out2, ws)
    torch.cuda.synchronize()
    assert optr.optr_device_error(p) == 0
    assert torch.equal(pool, pool2)
    assert win is None or torch.equal(win, win2)
    assert torch.equal(out, out2)
