"""A decode step on the tensor cores appends its own key and value rows: at the edges of the key
tile that holds them, with rows never written after them (NaN), over several layers, group sizes and
key-range splits.  The cache rows and positions are the CUDA-core route's (the suffix kernel's) bit
for bit; the outputs agree within both routes' rounding."""
import numpy as np
import pytest
import torch

import synth
from tests import _gpu_helpers as H

pytestmark = pytest.mark.gpu

L8B = synth.workload("llama8b")


def _steps(impl, wl, slots, steps, layer, split):
    """Decodes `steps` (per call, one index per request) after composing one chunk of slots[0] slots
    for each request; the cache's other rows hold NaN."""
    c2kv = H.lib()
    ctx = H.make_ctx(wl, pool_slots=max(slots) + 1, attn_impl=impl, attn_split=split)
    try:
        k, v = synth.chunk_slots(wl, 0, max(slots))
        assert len(set(slots)) == 1
        cid = c2kv.c2kv_compress_chunk(ctx, H.to_dev(k, wl), H.to_dev(v, wl), slots[0], 1, c2kv.MODE_STORED)
        ids = [cid] * len(slots)
        B, cap = len(slots), 1 + max(max(s) for s in steps)
        cache = c2kv.c2kv_compose(ctx, list(range(B + 1)), ids, None, cap)
        info = c2kv.c2kv_cache_info(cache)
        shp = (wl.layers, info["rows"], wl.n_kv_heads, wl.head_dim)
        ck, cv = (c2kv.device_view(info[x], shp, torch.bfloat16) for x in "kv")
        pos = c2kv.device_view(info["pos"], (info["rows"],), torch.int32)
        for b in range(B):
            end = int(info["row_base"][b] + info["n_slots"][b])
            last = int(info["row_base"][b] + info["capacity"][b])
            ck[:, end:last] = float("nan")
            cv[:, end:last] = float("nan")
            pos[end:last] = -1
        lq = wl.layers if layer < 0 else 1
        rng = np.random.default_rng(5)
        outs = []
        for st in steps:
            q = torch.from_numpy(rng.standard_normal((lq, B, wl.n_q_heads, 128), dtype=np.float32)).cuda().bfloat16()
            vn = torch.from_numpy(rng.standard_normal((lq, B, wl.n_kv_heads, 128), dtype=np.float32)).cuda().bfloat16()
            kn = q[:, :, ::wl.n_q_heads // wl.n_kv_heads].contiguous()   # its group's first query sees little else
            out = torch.full_like(q, float("nan"))
            lse = torch.full((lq, B, wl.n_q_heads), float("nan"), device="cuda")
            c2kv.c2kv_decode(ctx, cache, layer, q, kn, vn, st, out, lse)
            c2kv.c2kv_sync(ctx)
            outs.append((out.clone(), lse.clone()))
        rows = []
        for b in range(B):
            r0 = int(info["row_base"][b] + info["n_slots"][b])
            n = 1 + max(s[b] for s in steps)
            ls = slice(None) if layer < 0 else slice(layer, layer + 1)
            rows.append([x.clone() for x in (ck[ls, r0:r0 + n].float(), cv[ls, r0:r0 + n].float(), pos[r0:r0 + n])])
        return outs, rows
    finally:
        c2kv.c2kv_destroy(ctx)


@pytest.mark.parametrize("slots,count,split", [
    ([128], 2, 0),            # the new row opens a key tile, then follows itself
    ([127], 3, 0),            # the last row of a tile, then the next tile
    ([1], 2, 0),
    ([300, 300], 2, 3),       # splits: the last one appends, for each request
    ([1000], 2, 0),
    ([256], 2, 1), ([400], 2, 1), ([1000], 2, 1),   # 3, 4 and 8 tiles: the last one's stage used before
])
@pytest.mark.parametrize("hq,hkv,layers,layer", [(32, 8, 1, -1), (8, 1, 3, 1), (8, 8, 2, -1)])
def test_append(slots, count, split, hq, hkv, layers, layer):
    c2kv = H.lib()
    wl = synth.scaled(L8B, layers=layers, n_q_heads=hq, n_kv_heads=hkv)
    steps = [[i] * len(slots) for i in range(count)]
    tc, tc_rows = _steps(c2kv.ATTN_TC, wl, slots, steps, layer, split)
    cc, cc_rows = _steps(c2kv.ATTN_SIMT, wl, slots, steps, layer, 0)
    for (o, e), (o2, e2) in zip(tc, cc):
        assert torch.isfinite(o).all() and torch.isfinite(e).all()
        assert (o.float() - o2.float()).abs().max() <= 0.09   # 2^-9 of an outlier channel's 40, on either side
        assert (e - e2).abs().max() <= 1e-3
    for a, b in zip(tc_rows, cc_rows):
        for x, y in zip(a, b):
            assert torch.equal(x, y)


def test_append_zeroes_only_after_the_new_row():
    # a decode at index 3 zeroes up to its tile's edge once; the rows that later steps write stay
    c2kv = H.lib()
    wl = synth.scaled(L8B, layers=1)
    outs, rows = _steps(c2kv.ATTN_TC, wl, [100], [[0], [1], [2], [3], [2]], -1, 0)
    again, rows2 = _steps(c2kv.ATTN_SIMT, wl, [100], [[0], [1], [2], [3], [2]], -1, 0)
    for x, y in zip(rows[0], rows2[0]):
        assert torch.equal(x, y)
    assert torch.isfinite(outs[-1][0]).all()
