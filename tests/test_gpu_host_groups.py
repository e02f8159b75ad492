"""compose_attend over host-resident chunks in one to four layer groups (by the bytes that cross the
link), the last one short: the bits of compose, then attend, over the same chunks in the pool."""
import pytest
import torch

import synth
from tests import _gpu_helpers as H

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("layers,slots,sq", [
    (3, 640, 8),          # 8 MB: one group
    (5, 6000, 8),         # 123 MB: two groups, of three layers and two
    (7, 7000, 40),        # 212 MB: three groups, of three, three and one
    (9, 7000, 40),        # 273 MB: four groups, of three: the fourth has no layer left
])
def test_host_groups(layers, slots, sq):
    c2kv = H.lib()
    wl = synth.scaled(synth.workload("llama8b"), layers=layers, batch=1, chunk_tokens=slots, ratio_k=1, pool_chunks=1,
                      chunks_per_request=1, n_suffix=sq)
    gen = torch.Generator().manual_seed(3)
    kv = [torch.randn((layers, slots, wl.n_kv_heads, wl.head_dim), generator=gen).bfloat16().pin_memory() for _ in range(2)]
    q, k, v = (torch.randn((layers, 1, sq, h, wl.head_dim), generator=gen).bfloat16().cuda()
               for h in (wl.n_q_heads, wl.n_kv_heads, wl.n_kv_heads))
    outs = []
    for host in (True, False):
        ctx = H.make_ctx(wl, pool_slots=16 if host else slots, attn_split=1)
        try:
            src = kv if host else [x.cuda() for x in kv]
            cid = c2kv.c2kv_compress_chunk(ctx, *src, slots, 1, c2kv.MODE_HOST if host else c2kv.MODE_STORED)
            out = torch.full_like(q, float("nan"))
            lse = torch.full((layers, 1, wl.n_q_heads, sq), float("nan"), device="cuda")
            if host:
                cache = c2kv.c2kv_compose_attend(ctx, [0, 1], [cid], [5], sq, q, k, v, sq, out, lse)
            else:
                cache = c2kv.c2kv_compose(ctx, [0, 1], [cid], [5], sq)
                c2kv.c2kv_attend(ctx, cache, -1, q, k, v, sq, out, lse)
            c2kv.c2kv_sync(ctx)
            info = c2kv.c2kv_cache_info(cache)
            shp = (layers, info["rows"], wl.n_kv_heads, wl.head_dim)
            end = int(info["n_slots"][0]) + sq
            outs.append([out, lse] + [c2kv.device_view(info[x], shp, torch.bfloat16)[:, :end].clone() for x in "kv"])
        finally:
            c2kv.c2kv_destroy(ctx)
    assert not torch.isnan(outs[0][0]).any()
    for a, b in zip(*outs):
        assert torch.equal(a, b)
