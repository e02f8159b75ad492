"""How many query-tile pairs a CTA of the pair kernel runs in turn, or two CTAs of one tile an SM
(chosen by the rounds of CTAs that they save), does not change a bit of the result."""
import pytest
import torch

import synth
from tests import _gpu_helpers as H

pytestmark = pytest.mark.gpu

L8B = synth.scaled(synth.workload("llama8b"), layers=1, chunks_per_request=1)


@pytest.mark.parametrize("hq,batch,sq", [
    (32, 16, 128),     # 256 pairs: both of a head in turn
    (32, 24, 100),     # 384: one a CTA, the last with one part-full tile
    (64, 8, 120),      # 256, four a head: two in turn
    (32, 20, 200),     # 7 tiles a head, 640 pairs: 5 rounds; one tile a CTA, 4
])
def test_same_bits_for_any_number_in_turn(hq, batch, sq):
    c2kv = H.lib()
    wl = synth.scaled(L8B, n_q_heads=hq, batch=batch, chunk_tokens=1100, ratio_k=1, pool_chunks=1, n_suffix=sq)
    outs = []
    for pairs in (0, 1, 2):
        ctx = H.make_ctx(wl, pool_slots=1100, attn_pairs=pairs, attn_split=1)
        try:
            cid = c2kv.c2kv_compress_chunk(ctx, *(H.to_dev(x, wl) for x in synth.chunk_slots(wl, 0, 1100)), 1100, 1, c2kv.MODE_STORED)
            cache = c2kv.c2kv_compose(ctx, list(range(batch + 1)), [cid] * batch, [7 * r for r in range(batch)], sq)
            q, k, v = (H.to_dev(x, wl) for x in synth.suffix(wl))
            out = torch.full_like(q, float("nan"))
            lse = torch.full((1, batch, hq, sq), float("nan"), device="cuda")
            c2kv.c2kv_attend(ctx, cache, -1, q, k, v, sq, out, lse)
            c2kv.c2kv_sync(ctx)
            outs.append((out, lse))
        finally:
            c2kv.c2kv_destroy(ctx)
    assert not torch.isnan(outs[0][0]).any()
    for o, e in outs[1:]:
        assert torch.equal(outs[0][0], o) and torch.equal(outs[0][1], e)
