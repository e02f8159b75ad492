"""Compression at the edges of its work split: a thread's rows of one layer's block, or of several
layers when the ratio is small; a CTA's 256 items over parts of slots; the last slot's short block.
K within one storage ulp of the 64-bit mean turned to the slot's position, V bit-exact sums."""
import numpy as np
import pytest

import synth
from oracle import c2kv_oracle as orc
from tests import _gpu_helpers as H

pytestmark = pytest.mark.gpu

L8B = synth.workload("llama8b")
TINY = synth.workload("tiny_f32")


@pytest.mark.parametrize("base,hkv,d", [(L8B, 8, 128), (L8B, 1, 64), (L8B, 3, 128), (TINY, 2, 64), (TINY, 1, 128)])
@pytest.mark.parametrize("layers,n,k", [(1, 1, 1), (4, 37, 1), (5, 70, 1), (3, 71, 2), (2, 50, 3), (2, 301, 4), (3, 90, 7),
                                        (1, 200, 16), (1, 5, 9), (1, 71, 1), (1, 300, 1)])
def test_meanpool(base, hkv, d, layers, n, k):
    c2kv = H.lib()
    wl = synth.scaled(base, layers=layers, n_q_heads=4 * hkv, n_kv_heads=hkv, head_dim=d, chunk_tokens=n, ratio_k=k)
    kt, vt = synth.chunk_tokens(wl, 3)
    slots = orc.n_slots(n, k) + 5
    ctx = H.make_ctx(wl, pool_slots=slots)
    try:
        pad = c2kv.c2kv_compress_chunk(ctx, H.to_dev(kt[:, :1], wl), H.to_dev(vt[:, :1], wl), 1, 1, c2kv.MODE_MEANPOOL)
        cid = c2kv.c2kv_compress_chunk(ctx, H.to_dev(kt, wl), H.to_dev(vt, wl), n, k, c2kv.MODE_MEANPOOL)
        c2kv.c2kv_sync(ctx)
        gk, gv = H.pool_rows(ctx, wl, cid, slots)
        ok, ov = orc.compress_chunk(kt, vt, n, k, wl.rope_theta, wl.dtype, "meanpool")
        k_scale = orc.meanpool_slots(H.pair_magnitude(kt.astype(np.float64)), k)
        v_scale = orc.meanpool_slots(np.abs(vt.astype(np.float64)), k)
        H.check_rounded(gk, ok, k_scale, wl, "K")
        H.check_rounded(gv, ov, v_scale, wl, "V")
        assert c2kv.c2kv_chunk_info(ctx, pad)["slot_base"] == 0
    finally:
        c2kv.c2kv_destroy(ctx)


@pytest.mark.parametrize("layers,m", [(1, 1), (6, 33), (1, 33)])
def test_provided(layers, m):
    c2kv = H.lib()
    wl = synth.scaled(L8B, layers=layers, chunk_tokens=4 * m - 1, ratio_k=4)
    kb, vb = synth.chunk_slots(wl, 1, m)
    ctx = H.make_ctx(wl, pool_slots=m + 2)
    try:
        cid = c2kv.c2kv_compress_chunk(ctx, H.to_dev(kb, wl), H.to_dev(vb, wl), 4 * m - 1, 4, c2kv.MODE_PROVIDED)
        c2kv.c2kv_sync(ctx)
        gk, gv = H.pool_rows(ctx, wl, cid, m + 2)
        ok, ov = orc.compress_chunk(kb, vb, 4 * m - 1, 4, wl.rope_theta, wl.dtype, "provided")
        H.check_rotated(gk, ok, kb.astype(np.float64), wl, "provided K")
        assert np.array_equal(gv, vb.astype(np.float64))
    finally:
        c2kv.c2kv_destroy(ctx)
