"""A decode step that runs as a cache write and a decode (more than 256 new tokens,
CUDA-core variants) with pageable host memory for q or out is refused before the
write: pool, window store and output keep their bytes."""
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


@pytest.mark.parametrize("sink,recent", [(0, 0), (16, 48)])
@pytest.mark.parametrize("tokens,variants", [
    (300, {}),
    (3, dict(decode_variant=optr.OPTR_VARIANT_CUDA_CORE)),
    (3, dict(append_variant=optr.OPTR_VARIANT_CUDA_CORE)),
    (3, {}),
])
@pytest.mark.parametrize("pageable", ["q", "k", "v", "out"])
def test_pageable_memory_is_refused_before_the_cache_write(tokens, variants, sink, recent, pageable):
    h_kv = 2
    k, v = synth.kv_tokens(tokens, h_kv, "t4", 2, 0)
    R_k, R_v = synth.rotations(h_kv, 2)
    p = optr.optr_params_create(R_k, R_v, synth.key_mean(k), 4 * h_kv, sink=sink, recent=recent,
                                **variants)
    bt, pages = synth.page_tables([tokens], True, 2)
    i32 = lambda *x: torch.tensor(x, dtype=torch.int32, device="cuda")
    io = {"q": synth.queries(1, 4 * h_kv, 2), "k": k, "v": v, "out": torch.full((1, 4 * h_kv, 128), 7.0)}
    io = {n: x if n == pageable else x.cuda() for n, x in io.items()}
    pool = optr.new_pool(p, pages).fill_(0xA5)
    ws = optr.new_workspace(p, 1, bt.shape[1])
    args = (p, io["q"], io["k"], io["v"], i32(0, tokens), i32(0), bt.cuda(), i32(tokens), pool)
    win = optr.new_windows(p, 1).fill_(3.0) if sink else None
    with pytest.raises(ValueError):
        if sink:
            optr.optr_decode_step_win(*args, win, i32(0), io["out"], ws)
        else:
            optr.optr_decode_step(*args, io["out"], ws)
    torch.cuda.synchronize()
    assert (pool == 0xA5).all() and (io["out"] == 7.0).all()
    assert win is None or (win == 3.0).all()
