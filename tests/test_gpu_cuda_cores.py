"""The CUDA-core attention loop (fp32 contexts, and head layouts the tensor-core kernel does not
take) against the oracle: 16- and 64-row CTAs, one CTA a row tile and clusters of up to eight over
the keys, rows and keys at the edges of their tiles; the same loop under the extraction mask."""
import pytest

import synth
from tests.test_gpu_extract import _extract_case
from tests.test_gpu_parity import _attend_case

pytestmark = pytest.mark.gpu

F32 = synth.scaled(synth.workload("tiny_f32"), chunks_per_request=2, pool_chunks=2)
BF16 = synth.scaled(synth.workload("llama8b"), layers=1, chunks_per_request=2, pool_chunks=2)


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("hq,hkv,sq,tokens,k", [
    (1, 1, 1, 1, 1),         # one row, three keys
    (4, 2, 8, 28, 1),        # exactly one 16-row tile; 64 keys
    (4, 2, 9, 28, 1),        # two rows past it; one key past
    (6, 2, 43, 500, 4),      # G = 3, a ragged last tile
    (4, 1, 1, 2048, 1),      # few rows over 4096 keys: a cluster of eight
])
def test_attend_f32(d, hq, hkv, sq, tokens, k):
    _attend_case(synth.scaled(F32, n_q_heads=hq, n_kv_heads=hkv, head_dim=d, chunk_tokens=tokens, ratio_k=k), n_suffix=sq)


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("hq,hkv,sq", [(1, 1, 1), (4, 1, 1), (2, 1, 2), (2, 2, 4), (8, 2, 5), (3, 1, 2)])
@pytest.mark.parametrize("keys", [1, 8, 9, 16, 17, 32, 33, 64, 65, 200, 1100])
def test_attend_few_rows(d, hq, hkv, sq, keys):
    # four rows whose keys the warps share (key tiles partly full, warps without keys), and clusters of it
    if keys > sq:
        _attend_case(synth.scaled(F32, n_q_heads=hq, n_kv_heads=hkv, head_dim=d, chunk_tokens=keys - sq, ratio_k=1,
                                  chunks_per_request=1, pool_chunks=1), n_suffix=sq)


@pytest.mark.parametrize("d,sq,batch,hq,hkv", [(64, 250, 3, 32, 8), (128, 129, 4, 32, 8), (128, 16, 2, 64, 32)])
def test_attend_f32_large_launch(d, sq, batch, hq, hkv):
    # several CTAs per SM: 64 rows a CTA
    wl = synth.scaled(F32, n_q_heads=hq, n_kv_heads=hkv, head_dim=d, layers=2, batch=batch, chunk_tokens=300, ratio_k=4,
                      pool_chunks=2 * batch, draw="distinct")
    _attend_case(wl, n_suffix=sq)


@pytest.mark.parametrize("d,hq,hkv,impl", [(128, 6, 2, 0), (64, 6, 2, 0), (128, 8, 2, 1), (64, 32, 8, 1)])
def test_attend_bf16(d, hq, hkv, impl):
    # G = 3, and C2KV_ATTN_SIMT where the tensor cores would take the call
    _attend_case(synth.scaled(BF16, n_q_heads=hq, n_kv_heads=hkv, head_dim=d), n_suffix=45, attn_impl=impl)


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("n,k,layers", [(1, 1, 1), (63, 4, 2), (64, 1, 1), (130, 7, 1), (600, 16, 1), (333, 400, 1)])
def test_extract_f32(d, n, k, layers):
    _extract_case(synth.scaled(F32, head_dim=d), n, k, layers=layers)


@pytest.mark.parametrize("d", [64, 128])
def test_extract_group_of_three(d):
    _extract_case(synth.scaled(BF16, n_q_heads=24, n_kv_heads=8, head_dim=d), 260, 4, layers=2)
