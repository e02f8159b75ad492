"""Key-range splits chosen by the schedule that share SMs, two CTAs each, against the unsplit attend."""
import pytest
import torch

import synth
from tests import _gpu_helpers as H

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("hq,hkv,slots,sq", [
    (32, 8, [9000] * 3, 128),          # 96 query tiles of 72 key tiles: three splits
    (32, 8, [9000, 700, 6001], 100),   # ragged: a short request's later splits are empty
    (8, 8, [9000] * 2, 700),           # 96 tiles of 128 tokens
])
def test_shared_splits(hq, hkv, slots, sq):
    c2kv = H.lib()
    B = len(slots)
    wl = synth.scaled(synth.workload("llama8b"), layers=1, n_q_heads=hq, n_kv_heads=hkv, batch=B, chunk_tokens=max(slots),
                      ratio_k=1, pool_chunks=B, n_suffix=sq)
    outs = []
    for split in (0, 1):
        ctx = H.make_ctx(wl, pool_slots=sum(slots), attn_split=split)
        try:
            ids = []
            for i, n in enumerate(slots):
                k, v = synth.chunk_slots(wl, i, n)
                ids.append(c2kv.c2kv_compress_chunk(ctx, H.to_dev(k, wl), H.to_dev(v, wl), n, 1, c2kv.MODE_STORED))
            cache = c2kv.c2kv_compose(ctx, list(range(B + 1)), ids, None, sq)
            q, k, v = (H.to_dev(x, wl) for x in synth.suffix(wl))
            out = torch.full_like(q, float("nan"))
            lse = torch.full((1, B, hq, sq), float("nan"), device="cuda")
            c2kv.c2kv_profile_enable(ctx, True)
            c2kv.c2kv_attend(ctx, cache, -1, q, k, v, sq, out, lse)
            merges = c2kv.c2kv_profile_read(ctx)["combine"][1]
            info = c2kv.c2kv_cache_info(cache)
            cv = c2kv.device_view(info["v"], (1, info["rows"], hkv, wl.head_dim), torch.bfloat16)
            top = torch.stack([cv[:, int(r0):int(r0 + n) + sq].abs().amax(1) for r0, n in zip(info["row_base"], info["n_slots"])],
                              1).float()
            outs.append((out.float(), lse.clone(), merges))
        finally:
            c2kv.c2kv_destroy(ctx)
    (o, e, merges), (o2, e2, none) = outs
    assert (merges, none) == (1, 0)
    assert torch.isfinite(o).all() and torch.isfinite(e).all()
    # a split takes a weight against another maximum: its rounding to bf16 differs (2^-8 of it on either
    # side), and the output's (2^-8 on either side): 2^-6 of the channel's largest value
    assert ((o - o2).abs() <= 2.0 ** -6 * top.repeat_interleave(hq // hkv, dim=2)[:, :, None]).all()
    assert (e - e2).abs().max() <= 1e-4
