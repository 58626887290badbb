"""Sampling with top-k from the chunk maxima of the streaming kernel against the CPU oracle, at the edges of the chunks (32 or 64
vectors, 31 where rows start anywhere), of the bar (fewer chunks with a token than top_k, top_k beyond what takes a bar) and of the
list (more equal logits at the bar than it holds)."""
import numpy as np
import pytest

import synth
from synth import rng
from _gpu_util import Ctx
from test_gpu_sample_filtered import check_filtered, run_filtered

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("V,K,B", [(256, 9, 3), (257, 9, 33), (8191, 70, 31), (8192, 70, 9), (8193, 70, 67), (7936, 70, 5), (7945, 70, 130),
                                   (65536, 300, 600), (100003, 1500, 40), (128264, 2048, 65)])
def test_chunk_edges(V, K, B, dtype):
    if dtype == "f32" and B == 600:
        B = 300
    part = synth.zipf_partition(V, K, seed=V)
    cm = synth.class_mask_bernoulli(K, B, 0.3, rng.stream_key(rng.SEED_BASE, 930, V))
    cm[B // 2] = 0
    cm[B // 3] = 0
    cm[B // 3, 0] = 2  # one class
    z = synth.logits_normal(B, V, 2.0, dtype, (931, V))
    z[0, V - 1] = z[0].max()  # the largest logit also outside the vectors
    u = rng.uniform(rng.stream_key(932, V), B).astype(np.float32)
    with Ctx([part]) as ctx:
        for top_k, top_p in ((1, 1.0), (50, 0.9), (256, 1.0), (300, 0.95)):
            got = run_filtered(ctx, None, cm, z, V, u, 1.3, top_k, top_p)
            check_filtered(got, [part], None, cm, z, V, u, 1.3, top_k, top_p, "V=%d k=%d" % (V, top_k))


@pytest.mark.parametrize("B", [1, 31, 160])
def test_more_ties_at_the_bar_than_the_list_holds(B):
    V, K = 40000, 50
    part = synth.zipf_partition(V, K, seed=5)
    cm = synth.class_mask_bernoulli(K, B, 0.7, rng.stream_key(rng.SEED_BASE, 933))
    cm[:, 0] |= 1
    z = np.zeros((B, V), dtype=np.float32)
    z[:, ::1000] = 1.0
    u = rng.uniform(rng.stream_key(934), B).astype(np.float32)
    with Ctx([part]) as ctx:
        for top_k, top_p in ((100, 1.0), (100, 0.5)):
            got = run_filtered(ctx, None, cm, z, V, u, 1.0, top_k, top_p)
            check_filtered(got, [part], None, cm, z, V, u, 1.0, top_k, top_p, "k=%d p=%g" % (top_k, top_p))


def test_rows_of_several_partitions():
    V, B = 30001, 45
    parts = [synth.zipf_partition(V, k, seed=i) for i, k in enumerate((50, 333))]
    row_part = (np.arange(B) % 2).astype(np.int32)
    cm = synth.class_mask_bernoulli(333, B, 0.2, rng.stream_key(rng.SEED_BASE, 935))
    cm[:, 0] |= 1
    z = synth.logits_normal(B, V, 2.0, "bf16", (936,))
    u = rng.uniform(rng.stream_key(937), B).astype(np.float32)
    with Ctx(parts) as ctx:
        got = run_filtered(ctx, row_part, cm, z, V, u, 1.0, 50, 0.9)
        check_filtered(got, parts, row_part, cm, z, V, u, 1.0, 50, 0.9)


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
def test_every_vector_of_a_warp_holds_tokens_of_the_list(dtype):
    # 200 chunks with one token each that reaches the bar: the warps take four loads at a time, tokens in each of the four
    V, K, B = 65536, 40, 37
    part = synth.zipf_partition(V, K, seed=6)
    cm = synth.class_mask_bernoulli(K, B, 1.0, rng.stream_key(rng.SEED_BASE, 938))
    z = synth.logits_normal(B, V, 1.0, "f32", (939,))
    for b in range(B):
        z[b, np.arange(200) * 300 + (b * 7 + np.arange(200)) % 256] = 20.0 + np.arange(200) / 64.0
    if dtype == "bf16":
        z = (z.view(np.uint32) >> 16).astype(np.uint16)
    u = rng.uniform(rng.stream_key(940), B).astype(np.float32)
    with Ctx([part]) as ctx:
        for top_k, top_p in ((200, 1.0), (180, 0.9)):
            got = run_filtered(ctx, None, cm, z, V, u, 0.5, top_k, top_p)
            check_filtered(got, [part], None, cm, z, V, u, 0.5, top_k, top_p, "k=%d" % top_k)


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("V,B", [(253952, 3), (253961, 3), (256001, 1), (256001, 36), (262143, 2)])
def test_more_chunks_than_a_block_keeps(V, B, dtype):
    # rows off the vector grid have more than 1024 chunks from 253953 tokens on: the maxima past those count for the row's largest logit
    # and as chunks to read, and not for the bar
    K = 900
    part = synth.zipf_partition(V, K, seed=7)
    cm = synth.class_mask_bernoulli(K, B, 0.5, rng.stream_key(rng.SEED_BASE, 941, V))
    cm[:, 0] |= 1
    z = synth.logits_normal(B, V, 2.0, "f32", (942, V))
    allowed = synth.unpack_bits(cm, K)[:, part.c].astype(bool)
    for b in range(B):  # the row's keenest tokens among the last: the largest alone, then many
        last = np.flatnonzero(allowed[b, V - 2000:]) + V - 2000
        z[b, last[-1 - b % 7]] = 14.0
        if b % 2:
            z[b, last] = 12.0 + np.arange(len(last)) % 64 / 32.0
    if dtype == "bf16":
        z = (z.view(np.uint32) >> 16).astype(np.uint16)
    u = rng.uniform(rng.stream_key(943), B).astype(np.float32)
    with Ctx([part]) as ctx:
        for top_k, top_p in ((50, 0.9), (200, 1.0)):
            got = run_filtered(ctx, None, cm, z, V, u, 1.0, top_k, top_p)
            check_filtered(got, [part], None, cm, z, V, u, 1.0, top_k, top_p, "V=%d k=%d" % (V, top_k))
