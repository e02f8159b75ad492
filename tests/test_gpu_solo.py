"""The solo attention kernel (one query tile a CTA, alone on its SM or two sharing it, with and
without key-range splits and their merge launch) against the oracle and, where the split does not
change the order of sums, bit for bit against the pair kernel (attn_pairs = 1)."""
import pytest
import torch

import synth
from tests import _gpu_helpers as H
from tests.test_gpu_parity import _attend_case

pytestmark = pytest.mark.gpu

L8B = synth.scaled(synth.workload("llama8b"), layers=1, chunks_per_request=2, pool_chunks=2)


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("sq,tokens,k,batch", [
    (1, 64, 4, 1),         # one live token, one key tile
    (33, 256, 4, 2),       # the second query tile holds one token; 128 slots, then the suffix
    (20, 600, 1, 1),       # 10 key tiles: both S blocks and both K/V stages go round
])
def test_attend(d, sq, tokens, k, batch):
    _attend_case(synth.scaled(L8B, head_dim=d, chunk_tokens=tokens, ratio_k=k, batch=batch, pool_chunks=2 * batch,
                              draw="distinct"), n_suffix=sq)


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("sq,chunks", [(3, 2), (40, 4)])
def test_attend_splits_by_schedule(d, sq, chunks):
    # 2048-slot chunks, one request: the keys split over the SMs, the last split shorter
    _attend_case(synth.scaled(L8B, head_dim=d, chunk_tokens=2040, ratio_k=1, chunks_per_request=chunks,
                              pool_chunks=chunks), n_suffix=sq)


def test_attend_splits_of_unequal_requests():
    # the short request's later splits are empty
    wl = synth.scaled(L8B, chunk_tokens=2048, ratio_k=1, chunks_per_request=2, pool_chunks=2, n_kv_heads=2, n_q_heads=8,
                      batch=2)
    _attend_case(wl, requests=[([0, 1], [0, 2048]), ([1], [4])], n_suffix=10)


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("batch,sq,tokens", [
    (1, 40, 300),        # alone on its SM
    (8, 96, 256),        # 192 query tiles of 3 key tiles: two CTAs an SM
    (20, 30, 2200),      # one query tile per head, 160 of them: two CTAs an SM, 18 key tiles
])
def test_same_bits_as_the_pair_kernel(d, batch, sq, tokens):
    # (the larger launches against the pair kernel only: in the channels that carry 10 x N(0, 1) the
    # rounding of a weight to bf16 alone moves an output by up to 2^-9 x 40 = 0.08, which among 10^5
    # outputs exceeds the oracle comparison's 2e-2 now and then, with either kernel)
    c2kv = H.lib()
    wl = synth.scaled(L8B, head_dim=d, chunk_tokens=tokens, ratio_k=2, batch=batch, pool_chunks=4, n_suffix=sq)
    outs = []
    for pairs in (0, 1):
        ctx = H.make_ctx(wl, pool_slots=4 * tokens, attn_pairs=pairs, attn_split=1)
        try:
            ids = [c2kv.c2kv_compress_chunk(ctx, *(H.to_dev(x, wl) for x in synth.chunk_slots(wl, c, tokens // 2)), tokens, 2,
                                            c2kv.MODE_STORED) for c in range(4)]
            flat = [ids[(r + i) % 4] for r in range(batch) for i in range(2)]
            cache = c2kv.c2kv_compose(ctx, [2 * r for r in range(batch + 1)], flat, None, sq)
            q, k, v = (H.to_dev(x, wl) for x in synth.suffix(wl))
            out = torch.full_like(q, float("nan"))
            lse = torch.full((1, batch, wl.n_q_heads, sq), float("nan"), device="cuda")
            c2kv.c2kv_attend(ctx, cache, -1, q, k, v, sq, out, lse)
            c2kv.c2kv_sync(ctx)
            outs.append((out, lse))
        finally:
            c2kv.c2kv_destroy(ctx)
    assert not torch.isnan(outs[0][0]).any()
    assert torch.equal(outs[0][0], outs[1][0]) and torch.equal(outs[0][1], outs[1][1])


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("n,k,layers", [(33, 4, 1), (257, 8, 1), (1025, 16, 2)])
def test_extract_same_bits_as_the_pair_kernel(d, n, k, layers):
    c2kv = H.lib()
    wl = synth.scaled(L8B, n_q_heads=16, n_kv_heads=4, head_dim=d, layers=layers)
    q, kk, v = (H.to_dev(x, wl) for x in synth.extraction_inputs(wl, 0, n, k))
    outs = []
    for pairs in (0, 1):
        ctx = H.make_ctx(wl, pool_slots=64, attn_pairs=pairs)
        try:
            out = torch.full_like(q, float("nan"))
            lse = torch.full((layers, 16, q.shape[1]), float("nan"), device="cuda")
            c2kv.c2kv_extract_attention(ctx, layers, q, kk, v, n, k, out, lse)
            c2kv.c2kv_sync(ctx)
            outs.append((out, lse))
        finally:
            c2kv.c2kv_destroy(ctx)
    assert not torch.isnan(outs[0][0]).any()
    assert torch.equal(outs[0][0], outs[1][0]) and torch.equal(outs[0][1], outs[1][1])
