"""Decode steps of eight queries a KV head over more units than SMs: on the tensor cores, with weights of
two bf16 terms, against the CUDA-core kernel (fp32 weights) and the result in 64 bits."""
import numpy as np
import pytest
import torch

import synth
from tests import _gpu_helpers as H

pytestmark = pytest.mark.gpu

L8B = synth.workload("llama8b")


def _decode(impl, wl, slots, steps, q, kn, vn):
    c2kv = H.lib()
    B = len(steps)
    ctx = H.make_ctx(wl, pool_slots=slots, attn_impl=impl)
    try:
        k, v = synth.chunk_slots(wl, 0, slots)
        cid = c2kv.c2kv_compress_chunk(ctx, H.to_dev(k, wl), H.to_dev(v, wl), slots, 1, c2kv.MODE_STORED)
        cache = c2kv.c2kv_compose(ctx, list(range(B + 1)), [cid] * B, None, max(steps) + 1)
        info = c2kv.c2kv_cache_info(cache)
        shp = (wl.layers, info["rows"], wl.n_kv_heads, wl.head_dim)
        ck, cv = (c2kv.device_view(info[x], shp, torch.bfloat16) for x in "kv")
        gen = torch.Generator(device="cuda").manual_seed(1)
        for r0, n, cap in zip(info["row_base"], info["n_slots"], info["capacity"]):      # the earlier suffix rows
            for x in (ck, cv):
                x[:, int(r0 + n):int(r0 + cap)] = torch.randn(x[:, int(r0 + n):int(r0 + cap)].shape, generator=gen,
                                                              device="cuda").bfloat16()
        out = torch.full_like(q, float("nan"))
        lse = torch.full(q.shape[:3], float("nan"), device="cuda")
        c2kv.c2kv_profile_enable(ctx, True)
        c2kv.c2kv_decode(ctx, cache, -1, q, kn, vn, steps, out, lse)
        one_kernel = c2kv.c2kv_profile_read(ctx)["suffix"][1] == 0
        return out.double(), lse, one_kernel, [(ck[:, int(r0):int(r0 + n) + s + 1].double(), cv[:, int(r0):int(r0 + n) + s + 1].double())
                                               for r0, n, s in zip(info["row_base"], info["n_slots"], steps)]
    finally:
        c2kv.c2kv_destroy(ctx)


@pytest.mark.parametrize("layers,batch,slots", [(1, 20, 257), (1, 20, 380), (5, 4, 1000), (1, 40, 2300)])
def test_two_terms(layers, batch, slots):
    c2kv = H.lib()
    wl = synth.scaled(L8B, layers=layers, n_q_heads=64, n_kv_heads=8)
    gen = torch.Generator(device="cuda").manual_seed(2)
    q, kn, vn = (2 * torch.randn((layers, batch, h, 128), generator=gen, device="cuda").bfloat16() for h in (64, 8, 8))
    steps = [(7 * b) % 5 for b in range(batch)]
    o, e, one_kernel, rows = _decode(0, wl, slots, steps, q, kn, vn)
    o2, e2, two_kernels, rows2 = _decode(c2kv.ATTN_SIMT, wl, slots, steps, q, kn, vn)
    assert one_kernel and not two_kernels
    worst, worst2 = 0.0, 0.0
    for b, ((k, v), (k2, v2)) in enumerate(zip(rows, rows2)):
        assert torch.equal(k, k2) and torch.equal(v, v2)
        # in 64 bits, from the turned rows; the queries turned as the key of the same position is
        pos = slots + steps[b]
        i = torch.arange(64, device="cuda", dtype=torch.float64)
        ang = pos * wl.rope_theta ** (-i / 64)
        c, s = torch.cos(ang), torch.sin(ang)
        x, y = q[:, b, :, :64].double(), q[:, b, :, 64:].double()
        qr = torch.cat([x * c - y * s, y * c + x * s], -1).bfloat16().double()
        sc = torch.einsum("lhgd,lnhd->lhgn", qr.view(layers, 8, 8, 128), k) / np.sqrt(128.0)
        want = torch.einsum("lhgn,lnhd->lhgd", torch.softmax(sc, -1), v).reshape(layers, 64, 128)
        # an output's rounding to bf16 on either side (8 significant bits: half a unit is up to 2^-8 of
        # the value, so 2^-7 together), and the weights' second rounding (2^-8 of 2^-8)
        top = v.abs().amax(1).repeat_interleave(8, 1)
        assert ((o[:, b] - o2[:, b]).abs() <= 2.0 ** -7 * o2[:, b].abs() + 2.0 ** -16 * top).all()
        worst = max(worst, float(((o[:, b] - want) ** 2).sum()))
        worst2 = max(worst2, float(((o2[:, b] - want) ** 2).sum()))
    assert (e - e2).abs().max() <= 1e-5 * e2.abs().max()
    assert worst <= 1.02 * worst2      # both dominated by the output's rounding
