"""compose_attend composes first, then attends, when ragged chunks leave most key tiles with a
boundary; it stays fused when every tile lies in one chunk.  Either way the bits of the other route."""
import pytest
import torch

import synth
from tests import _gpu_helpers as H

pytestmark = pytest.mark.gpu

L8B = synth.workload("llama8b")


@pytest.mark.parametrize("layers,batch,slots,count,sq,want_fused", [
    (2, 2, 125, 6, 64, False),     # a boundary in every tile
    (2, 1, 128, 3, 64, True),      # none
    (1, 8, 500, 3, 30, False),     # in three tiles of twelve; one query tile a head
    (4, 1, 250, 1, 64, False),     # one chunk: the suffix's boundary alone
    (1, 1, 131, 1, 1, False),
])
def test_route_and_bits(layers, batch, slots, count, sq, want_fused):
    c2kv = H.lib()
    wl = synth.scaled(L8B, layers=layers, batch=batch, chunk_tokens=slots, ratio_k=1, pool_chunks=1, n_suffix=sq)
    outs, fused = [], []
    for fuse in (0, c2kv.FUSE_ALWAYS):
        ctx = H.make_ctx(wl, pool_slots=slots, fuse=fuse, attn_split=1)
        try:
            cid = c2kv.c2kv_compress_chunk(ctx, *(H.to_dev(x, wl) for x in synth.chunk_slots(wl, 0, slots)), slots, 1,
                                           c2kv.MODE_STORED)
            q, k, v = (H.to_dev(x, wl) for x in synth.suffix(wl, layers=layers))
            out = torch.full_like(q, float("nan"))
            lse = torch.full((layers, batch, wl.n_q_heads, sq), float("nan"), device="cuda")
            args = ([count * r for r in range(batch + 1)], [cid] * (count * batch),
                    [slots * i for _ in range(batch) for i in range(count)], sq, q, k, v, sq, out, lse)
            c2kv.c2kv_profile_enable(ctx, True)
            cache = c2kv.c2kv_compose_attend(ctx, *args)
            fused.append(c2kv.c2kv_profile_read(ctx)["fused"][1] == 1)
            c2kv.c2kv_profile_enable(ctx, False)
            c2kv.c2kv_cache_release(ctx, cache)
            out.fill_(float("nan"))
            cache = c2kv.c2kv_compose_attend(ctx, *args)      # untraced: the overlapped route
            c2kv.c2kv_sync(ctx)
            info = c2kv.c2kv_cache_info(cache)
            shp = (layers, info["rows"], wl.n_kv_heads, wl.head_dim)
            kv = [c2kv.device_view(info[x], shp, torch.bfloat16) for x in "kv"]
            ends = [(int(r0), int(r0 + n) + sq) for r0, n in zip(info["row_base"], info["n_slots"])]
            outs.append([out, lse] + [x[:, a:b].clone() for x in kv for a, b in ends])
        finally:
            c2kv.c2kv_destroy(ctx)
    assert fused == [want_fused, True]
    assert not torch.isnan(outs[0][0]).any()
    for a, b in zip(*outs):
        assert torch.equal(a, b)
