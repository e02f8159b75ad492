"""Decode steps of eight queries a KV head over more units than SMs: on the tensor cores, with fp32 weights
in three bf16 terms, against the CUDA-core kernel (fp32 weights) and the result in 64 bits."""
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
def test_terms(layers, batch, slots):
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
        # the value, so 2^-7 together), and the sums' errors, far below 2^-16 of the largest value
        top = v.abs().amax(1).repeat_interleave(8, 1)
        assert ((o[:, b] - o2[:, b]).abs() <= 2.0 ** -7 * o2[:, b].abs() + 2.0 ** -16 * top).all()
        worst = max(worst, float(((o[:, b] - want) ** 2).sum()))
        worst2 = max(worst2, float(((o2[:, b] - want) ** 2).sum()))
    assert (e - e2).abs().max() <= 1e-5 * e2.abs().max()
    assert worst <= 1.02 * worst2      # both dominated by the output's rounding


def _both_routes(wl, fill, slots, steps, suffix=None):
    """Decodes a token of zero key and value over a cache that fill(ck, cv, info) sets, on the automatic
    route and on the CUDA cores; suffix: rows (k, v) that an attend call writes before."""
    c2kv = H.lib()
    B = len(steps)
    gen = torch.Generator(device="cuda").manual_seed(4)
    q = torch.randn((wl.layers, B, wl.n_q_heads, 128), generator=gen, device="cuda").bfloat16()
    zero = torch.zeros((wl.layers, B, wl.n_kv_heads, 128), device="cuda").bfloat16()
    got = []
    for impl in (c2kv.ATTN_AUTO, c2kv.ATTN_SIMT):
        ctx = H.make_ctx(wl, pool_slots=slots, attn_impl=impl)
        try:
            rows = torch.zeros((wl.layers, slots, wl.n_kv_heads, 128), device="cuda").bfloat16()
            cid = c2kv.c2kv_compress_chunk(ctx, rows, rows, slots, 1, c2kv.MODE_STORED)
            n = 0 if suffix is None else suffix[0].shape[2]
            cache = c2kv.c2kv_compose(ctx, list(range(B + 1)), [cid] * B, None, max(n, max(steps) + 1))
            if n:
                qs = torch.zeros((wl.layers, B, n, wl.n_q_heads, 128), device="cuda").bfloat16()
                c2kv.c2kv_attend(ctx, cache, -1, qs, *suffix, n, torch.empty_like(qs))
            info = c2kv.c2kv_cache_info(cache)
            shp = (wl.layers, info["rows"], wl.n_kv_heads, 128)
            fill(*(c2kv.device_view(info[x], shp, torch.bfloat16) for x in "kv"), info)
            out = torch.full_like(q, float("nan"))
            c2kv.c2kv_profile_enable(ctx, True)
            c2kv.c2kv_decode(ctx, cache, -1, q, zero, zero, steps, out)
            assert (c2kv.c2kv_profile_read(ctx)["suffix"][1] == 0) == (impl == c2kv.ATTN_AUTO)
            got.append(out.double())
        finally:
            c2kv.c2kv_destroy(ctx)
    return got


@pytest.mark.parametrize("layers,batch,slots", [(1, 20, 300), (20, 1, 600)])
def test_weights_hold_fp32(layers, batch, slots):
    """As tests/test_gpu_heads64.py: two keys of values 1 and -1 whose weights differ by some 2^-14, among
    keys of score and value 0.  A rounding flip of the output (up to 2^-7 of it), and two exponentials of error
    2^-22 on either route over a sum of at least half of `slots`; 16-bit weights are off by up to 2^-17."""
    wl = synth.scaled(L8B, layers=layers, n_q_heads=64, n_kv_heads=8)
    gen = torch.Generator(device="cuda").manual_seed(5)
    key = 0.1 * torch.randn((layers, 8, 128), generator=gen, device="cuda")      # scores near 0, all weights near 1

    def fill(ck, cv, info):
        for r0 in info["row_base"]:
            for i, (c0, v) in enumerate([(0.0, 1.0), (2.0 ** -11, -1.0)]):
                key[..., 0] = c0
                ck[:, int(r0) + i] = key.bfloat16()
                cv[:, int(r0) + i] = v

    o, o2 = _both_routes(wl, fill, slots, [0] * batch)
    over = (o - o2).abs() - (2.0 ** -7 * o2.abs() + 2.0 ** -20 / (slots / 2))
    assert (over <= 0).all(), f"{float((over > 0).double().mean()):.3f} of the outputs off by up to {float(over.max()):.3g} more"


def test_infinite_values():
    """A visible value of plus or minus infinity gives it (both: NaN); rows after the new one, written by an
    earlier attend call, do not count whatever they hold."""
    wl = synth.scaled(L8B, layers=20, n_q_heads=64, n_kv_heads=8)
    inf = float("inf")
    ks = torch.zeros((20, 1, 4, 8, 128), device="cuda").bfloat16()
    vs = ks.clone()
    vs[:, :, 2:] = torch.tensor([inf, float("nan")], device="cuda").view(1, 1, 2, 1, 1)

    def fill(ck, cv, info):
        r0 = int(info["row_base"][0])
        cv[:, r0:r0 + 380] = 1.0
        cv[:, r0 + 3, :, 0] = inf
        cv[:, r0 + 301, :, 1] = -inf
        cv[:, r0 + 3, :, 2], cv[:, r0 + 200, :, 2] = inf, -inf

    o, o2 = _both_routes(wl, fill, 380, [1], (ks, vs))
    assert (o2[..., 0] == inf).all() and (o2[..., 1] == -inf).all() and o2[..., 2].isnan().all()
    assert o2[..., 3:].isfinite().all()
    assert torch.equal(o[..., :3].nan_to_num(7.0), o2[..., :3].nan_to_num(7.0))
    assert ((o - o2)[..., 3:].abs() <= 2.0 ** -7).all()
