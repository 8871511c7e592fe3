"""Long cache writes against the same tokens written a little at a time.

A CTA of the tensor-core cache write passes its tiles through rings of stages,
A operands, accumulators and record places.  One call with many tiles per CTA
has to give the bytes that calls with one or two tiles per CTA give, at whole and
ragged tile counts, one and two epilogue groups, both records.
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


@pytest.mark.parametrize("group,clip", [(32, 1.0), (128, 0.95)])
@pytest.mark.parametrize("h_kv,tokens", [
    (8, 9 * 128 * 9),           # 9 tiles per CTA: one more than the places kept
    (8, 9 * 128 * 16 + 1),      # 16 and 17
    (16, 4 * 128 * 33 - 5),     # 33, the last one ragged
    (19, 4 * 128 * 5 + 77),     # 4 CTAs of 5 or 6
])
def test_long_write_is_its_short_writes(group, clip, h_kv, tokens):
    k, v = synth.kv_tokens(tokens, h_kv, "t4", 11, 0)
    R_k, R_v = synth.rotations(h_kv, 11)
    p = optr.optr_params_create(R_k, R_v, synth.key_mean(k), 4 * h_kv, clip_k=clip, clip_v=clip,
                                group=group)
    bt, pages = synth.page_tables([tokens], True, 11)
    k, v, bt = k.cuda(), v.cuda(), bt.cuda()
    pools = [optr.new_pool(p, pages) for _ in range(2)]
    for pool, step in zip(pools, (tokens, 512)):
        for t in range(0, tokens - step + 1, step):
            n = step if t + 2 * step <= tokens else tokens - t  # (no short rest)
            optr.optr_kv_append(p, k[t:t + n], v[t:t + n],
                                torch.tensor([0, n], dtype=torch.int32, device="cuda"),
                                torch.tensor([t], dtype=torch.int32, device="cuda"), bt, pool)
    torch.cuda.synchronize()
    assert optr.optr_device_error(p) == 0
    assert torch.equal(*pools)
