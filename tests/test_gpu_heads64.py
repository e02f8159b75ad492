"""bf16 heads of 64 channels on the tensor cores: the suffix attention and the extraction
attention against the oracle and against the CUDA-core kernel, at the edges of the query and key
tiles (128 packed rows, 128 keys), over the group sizes and key-range splits."""
import os
import subprocess
import sys

import numpy as np
import pytest
import torch

import synth
from tests import _gpu_helpers as H
from tests.test_gpu_extract import _extract_case
from tests.test_gpu_parity import _attend_case
from tests.test_zz_no_alloc import _FIRST_CALL

pytestmark = pytest.mark.gpu

D64 = synth.scaled(synth.workload("llama8b"), layers=1, head_dim=64, chunks_per_request=2, pool_chunks=2)


@pytest.mark.parametrize("hq,hkv,sq,tokens,k", [
    (4, 1, 1, 64, 1),        # one row tile, keys end one past a tile (2 x 64 slots + 1)
    (4, 1, 32, 256, 4),      # exactly one 128-row tile
    (4, 1, 33, 252, 4),      # one token past it
    (8, 2, 64, 300, 10),     # exactly a pair of tiles
    (8, 2, 65, 300, 10),     # a second pair of one token
    (2, 2, 129, 64, 4),      # G = 1: a tile past one pair's half
    (32, 2, 17, 97, 16),     # G = 16: eight tokens a tile
    (16, 2, 47, 2048, 1),    # 4096 slots, G = 8
])
def test_attend(hq, hkv, sq, tokens, k):
    _attend_case(synth.scaled(D64, n_q_heads=hq, n_kv_heads=hkv, chunk_tokens=tokens, ratio_k=k), n_suffix=sq)


@pytest.mark.parametrize("hq,hkv,sq,tokens,k", [(4, 1, 1, 64, 1), (8, 2, 3, 20, 4), (1, 1, 4, 1, 1), (32, 8, 1, 150, 1)])
def test_attend_short(hq, hkv, sq, tokens, k):
    # few rows over few keys: on the tensor cores when splits are asked for, else on the CUDA cores
    wl = synth.scaled(D64, n_q_heads=hq, n_kv_heads=hkv, chunk_tokens=tokens, ratio_k=k)
    _attend_case(wl, n_suffix=sq, attn_split=1)
    _attend_case(synth.scaled(wl, layers=24), n_suffix=sq)


@pytest.mark.parametrize("n_suffix", [1, 48])
def test_noalloc_first_call_takes_no_device_memory(n_suffix):
    # either route's kernels are loaded when the context is made
    script = _FIRST_CALL.replace("n_suffix=16)", f"n_suffix={n_suffix}, head_dim=64, chunk_tokens=64)")
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    res = subprocess.run([sys.executable, "-c", script.format(root=root)], env=dict(os.environ, CUDA_MODULE_LOADING="LAZY"),
                         capture_output=True, text=True, timeout=240, cwd=root)
    assert res.returncode == 0, res.stdout[-2000:] + res.stderr[-2000:]
    assert "FREE_DELTA 0\n" in res.stdout, res.stdout[-2000:]


@pytest.mark.parametrize("split", [2, 5, 16])
def test_attend_splits(split):
    # three key tiles: with more splits some are empty, and they merge in the kernel
    _attend_case(synth.scaled(D64, chunk_tokens=64, chunks_per_request=1, pool_chunks=1), n_suffix=300,
                 attn_split=split)


def test_attend_layer_of_a_batch():
    wl = synth.scaled(synth.workload("batched"), head_dim=64, layers=3, batch=3, chunks_per_request=4,
                      pool_chunks=32, n_suffix=70)
    _attend_case(wl, layer=1)


@pytest.mark.parametrize("n,k", [(512, 4), (128, 1), (129, 16), (33, 4), (1, 1), (700, 10)])
def test_extract(n, k):
    # (short chunks: on the CUDA cores by themselves, on the tensor cores with pairs that are asked for)
    _extract_case(D64, n, k, layers=2 if n < 200 else 1)
    if n < 200:
        _extract_case(D64, n, k, layers=2, attn_pairs=1)
        _extract_case(D64, n, k, layers=40 if n > 1 else 2)


def test_weights_keep_more_than_bf16():
    """The tensor-core kernel's output is off the CUDA-core kernel's by at most a rounding flip of the
    bf16 output (2^-8 of the value) and, per unit weight, 2^-15 of the largest value.  Weights of one
    bf16 term would be off by 2^-9 of it."""
    c2kv = H.lib()
    wl = synth.scaled(D64, n_suffix=50, chunks_per_request=4, pool_chunks=4)
    (ids, offs), = synth.requests(wl)
    chunks = H.oracle_chunks_meanpool(wl, ids)
    q, ks, vs = (H.to_dev(x, wl) for x in synth.suffix(wl))
    outs = []
    for impl in (c2kv.ATTN_AUTO, c2kv.ATTN_SIMT):
        ctx = H.make_ctx(wl, pool_slots=4 * 128 + 16, attn_impl=impl)
        try:
            dev = H.load_stored(ctx, wl, chunks)
            cache = c2kv.c2kv_compose(ctx, [0, len(ids)], [dev[c] for c in ids], offs, suffix_capacity=50)
            out = torch.full_like(q, float("nan"))
            c2kv.c2kv_attend(ctx, cache, -1, q, ks, vs, 50, out)
            c2kv.c2kv_sync(ctx)
            outs.append(out.double().cpu().numpy())
        finally:
            c2kv.c2kv_destroy(ctx)
    vmax = max(float(vs.abs().max()), max(float(np.abs(c[1]).max()) for c in chunks.values()))
    allowed = 2.0 ** -8 * np.abs(outs[1]) + 4 * 2.0 ** -17 * vmax
    assert (np.abs(outs[0] - outs[1]) <= allowed).all(), float((np.abs(outs[0] - outs[1]) - allowed).max())


@pytest.mark.parametrize("layers,pairs", [(16, 0), (80, 0), (16, 1)], ids=["alone", "shared", "pair"])
def test_weights_hold_fp32(layers, pairs):
    """Two keys that differ by a little in one channel and carry values 1 and -1: the output is the
    difference of their weights, some 2^-14 of either.  The CUDA-core kernel's weights are fp32, and both
    routes read the same turned queries and cached rows, so what may differ is a rounding flip of the
    output (a unit of 8 significant bits, up to 2^-7 of it) and two exponentials, of error 2^-22 each, on
    either route: 2^-20 for weights of at most 1 over a sum of at least 1.  Weights of 16 significant bits
    are off by up to 2^-17 each."""
    c2kv = H.lib()
    n = 32
    wl = synth.scaled(D64, n_q_heads=8, n_kv_heads=2, layers=layers)
    gen = torch.Generator(device="cuda").manual_seed(3)
    q = torch.randn((layers, 1, n, 8, 64), generator=gen, device="cuda").bfloat16()
    zero = torch.zeros((layers, 1, n, 2, 64), device="cuda").bfloat16()       # suffix rows: score 0, value 0
    rows = torch.randn((layers, 1, 2, 64), generator=gen, device="cuda").repeat(1, 2, 1, 1)
    rows[..., 0] = torch.tensor([0.0, 2.0 ** -11], device="cuda").view(1, 2, 1)
    outs = []
    for impl in (c2kv.ATTN_AUTO, c2kv.ATTN_SIMT):
        ctx = H.make_ctx(wl, pool_slots=2, attn_impl=impl, attn_pairs=pairs)
        try:
            cid = c2kv.c2kv_compress_chunk(ctx, rows.bfloat16(), rows.bfloat16(), 2, 1, c2kv.MODE_STORED)
            cache = c2kv.c2kv_compose(ctx, [0, 1], [cid], None, suffix_capacity=n)
            info = c2kv.c2kv_cache_info(cache)
            ck, cv = (c2kv.device_view(info[x], (layers, info["rows"], 2, 64), torch.bfloat16) for x in "kv")
            ck[:, :2] = rows.bfloat16()
            cv[:, 0], cv[:, 1] = 1.0, -1.0
            out = torch.full_like(q, float("nan"))
            c2kv.c2kv_attend(ctx, cache, -1, q, zero, zero, n, out)
            c2kv.c2kv_sync(ctx)
            outs.append(out.double())
        finally:
            c2kv.c2kv_destroy(ctx)
    over = (outs[0] - outs[1]).abs() - (2.0 ** -7 * outs[1].abs() + 2.0 ** -20)
    assert (over <= 0).all(), f"{float((over > 0).double().mean()):.3f} of the outputs off by up to {float(over.max()):.3g} more"


def test_forced_tensor_cores_stay_refused():
    c2kv = H.lib()
    with pytest.raises(c2kv.C2KVError) as e:
        H.make_ctx(D64, pool_slots=64, attn_impl=c2kv.ATTN_TC)
    assert e.value.status == c2kv.ERR_UNSUPPORTED
