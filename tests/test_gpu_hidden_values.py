"""Values of infinity and NaN in rows that some queries see and others do not: a row's output depends on the
rows it sees only.  Each call runs on finite values and again with some of them replaced; the queries that do
not see those rows give the same result, the others what the sums give."""
import pytest
import torch

import synth
from tests import _gpu_helpers as H

pytestmark = pytest.mark.gpu

INF, NAN = float("inf"), float("nan")
# (dtype, d, Hq, Hkv): the CUDA cores' loop, one CTA a row tile and clusters
CUDA_CORES = [("f32", 64, 4, 2), ("f32", 128, 16, 4), ("bf16", 64, 6, 2), ("bf16", 128, 6, 2)]


def _rand(seed, *shape):
    return torch.randn(shape, generator=torch.Generator(device="cuda").manual_seed(seed), device="cuda")


def _same(a, b, bits):
    """Finite and the same: bit for bit, or (one of them from another kernel) within both sides' rounding
    to bf16, 2^-7 of the value, and the sums' errors."""
    if bits:
        return torch.equal(a, b) and bool(a.isfinite().all())
    a, b = a.double(), b.double()
    return bool(((a - b).abs() <= 2.0 ** -7 * b.abs() + 2.0 ** -12).all())


def _attend(wl, slots, n, spoil, layers, split, pairs):
    c2kv = H.lib()
    td = H.tdtype(wl)
    hq, hkv, d = wl.n_q_heads, wl.n_kv_heads, wl.head_dim
    k, v = (_rand(i, layers, slots, hkv, d).to(td) for i in (1, 2))
    q, ks, vs = (_rand(i, layers, 1, n, h, d).to(td) for i, h in ((3, hq), (4, hkv), (5, hkv)))
    spoil(v, vs)
    ctx = H.make_ctx(synth.scaled(wl, layers=layers), pool_slots=slots, attn_split=split, attn_pairs=pairs)
    try:
        cid = c2kv.c2kv_compress_chunk(ctx, k, v, slots, 1, c2kv.MODE_STORED)
        cache = c2kv.c2kv_compose(ctx, [0, 1], [cid], None, suffix_capacity=n)
        out, lse = torch.full_like(q, 7.0), torch.zeros((layers, 1, hq, n), device="cuda")
        c2kv.c2kv_attend(ctx, cache, -1, q, ks, vs, n, out, lse)
        c2kv.c2kv_sync(ctx)
        return out[:, 0], lse
    finally:
        c2kv.c2kv_destroy(ctx)


def check_attend(dtype, d, hq, hkv, slots=200, n=90, layers=1, split=1, pairs=0, bits=True):
    wl = synth.scaled(synth.workload("tiny_f32" if dtype == "f32" else "llama8b"), n_q_heads=hq, n_kv_heads=hkv, head_dim=d)

    def run(spoil):
        return _attend(wl, slots, n, spoil, layers, split, pairs)

    def late(v, vs):                 # two of the last tokens' values
        vs[:, 0, n - 3, :, :] = INF
        vs[:, 0, n - 1, :, 1] = NAN

    def seen(v, vs):                 # a composed slot's, which every query sees
        v[:, 5, :, 2], v[:, 6, :, 3] = -INF, INF
        v[:, 7, :, 4], v[:, slots - 1, :, 4] = INF, -INF

    clean, lse = run(lambda v, vs: None)
    out, lse1 = run(late)
    assert _same(out[:, :n - 3], clean[:, :n - 3], bits)
    assert (out[:, n - 3:n - 1] == INF).all() and (out[:, n - 1, :, 2:] == INF).all() and out[:, n - 1, :, 1].isnan().all()
    out, lse2 = run(seen)
    assert (out[..., 2] == -INF).all() and (out[..., 3] == INF).all() and out[..., 4].isnan().all()
    keep = [c for c in range(d) if c not in (2, 3, 4)]
    assert _same(out[..., keep], clean[..., keep], bits)
    assert torch.equal(lse, lse1) and torch.equal(lse, lse2)


def check_extract(dtype, d, hq, hkv, n, k, bits=True, pairs=0, layers=1):
    c2kv = H.lib()
    wl = synth.scaled(synth.workload("tiny_f32" if dtype == "f32" else "llama8b"), n_q_heads=hq, n_kv_heads=hkv, head_dim=d)
    m = -(-n // k)
    t0 = n - k - 2                                    # a document token of the last block but one

    def run(spoil):
        q, kk, v = (_rand(i, layers, n + m, h, d).to(H.tdtype(wl)) for i, h in ((1, hq), (2, hkv), (3, hkv)))
        if spoil:
            v[:, t0] = INF
            v[:, n + m - 2] = NAN                     # and a C2 token
        out, lse = torch.full_like(q, 7.0), torch.zeros((layers, hq, n + m), device="cuda")
        ctx = H.make_ctx(wl, pool_slots=16, attn_pairs=pairs)
        try:
            c2kv.c2kv_extract_attention(ctx, layers, q, kk, v, n, k, out, lse)
            c2kv.c2kv_sync(ctx)
        finally:
            c2kv.c2kv_destroy(ctx)
        return out, lse

    clean, lse = run(False)
    out, lse2 = run(True)
    j = t0 // k                                       # c_j sees the token; c_(m-2) and c_(m-1) the other
    assert _same(out[:, :t0], clean[:, :t0], bits) and (out[:, t0:n] == INF).all()
    for c in range(m):
        o = out[:, n + c]
        if c >= m - 2:
            assert o.isnan().all(), c
        elif c == j:
            assert (o == INF).all(), c
        else:
            assert _same(o, clean[:, n + c], bits), c
    assert torch.equal(lse, lse2)


@pytest.mark.parametrize("dtype,d,hq,hkv", CUDA_CORES)
def test_attend(dtype, d, hq, hkv):
    check_attend(dtype, d, hq, hkv)


@pytest.mark.parametrize("dtype,d,hq,hkv", CUDA_CORES)
def test_attend_large(dtype, d, hq, hkv):
    check_attend(dtype, d, hq, hkv, slots=100, n=200, layers=24)      # 64 rows a CTA, no cluster


@pytest.mark.parametrize("dtype,d,hq,hkv", CUDA_CORES)
@pytest.mark.parametrize("n,k", [(150, 4), (333, 16)])
def test_extract(dtype, d, hq, hkv, n, k):
    check_extract(dtype, d, hq, hkv, n, k)


# bf16 heads of 64 channels on the tensor cores, in each form of the kernel
@pytest.mark.parametrize("hq,hkv", [(32, 8), (16, 16), (32, 4)])
@pytest.mark.parametrize("form", [dict(), dict(layers=30), dict(pairs=1), dict(split=3), dict(pairs=2, n=200), dict(split=0, slots=2500)],
                         ids=["alone", "shared", "pair", "merged", "pairs_in_turn", "split"])
def test_attend_heads64(hq, hkv, form):
    check_attend("bf16", 64, hq, hkv, bits=False, **form)


@pytest.mark.parametrize("hq,hkv", [(32, 8), (16, 16)])
@pytest.mark.parametrize("n,k,pairs", [(150, 4, 0), (333, 16, 0), (333, 16, 1)])
def test_extract_heads64(hq, hkv, n, k, pairs):
    check_extract("bf16", 64, hq, hkv, n, k, bits=False, pairs=pairs, layers=2)
