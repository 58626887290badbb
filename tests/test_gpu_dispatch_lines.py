"""Calls on either side of the lines at which a step takes another kernel, against the CPU oracle: rows that allow few tokens
(row count, classes, row length, mixed batches) and several masks per row (masks, classes, row length)."""
import numpy as np
import pytest

import synth
import test_gpu_multi_mask
from synth import rng
from paper_2605_29986_b200 import binding as cz
from _gpu_util import Ctx, compare_step, oracle_step, run_fused

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("V,K,B,parts", [
    (9000, 300, 63, 1), (9000, 300, 64, 1),
    (60000, 4800, 64, 1), (60000, 5100, 64, 1), (60000, 16000, 64, 1),       # masks in slices of 128 words; two blocks per SM, one
    (9000, 200, 296, 1), (9000, 200, 297, 1), (60000, 200, 444, 1), (60000, 200, 445, 1), (60000, 200, 593, 1),
    (20000, 3072, 64, 2), (20000, 3080, 64, 2), (9000, 200, 63, 3), (9000, 200, 420, 3), (9000, 200, 500, 4)])
def test_rows_that_allow_few_tokens(V, K, B, parts, dtype):
    ps = [synth.zipf_partition(V, K, seed=80 + i) for i in range(parts)]
    row_part = None if parts == 1 else (np.arange(B) * 5 % parts).astype(np.int32)
    cm = synth.class_mask_bernoulli(K, B, 0.01, rng.stream_key(rng.SEED_BASE, 911, V, K))
    cm[:, 0] |= 2
    z = synth.logits_normal(B, V, 2.0, dtype, (912, V, K))
    with Ctx(ps) as ctx:
        compare_step(run_fused(ctx, row_part, cm, z, V, mode=cz.SPARSE), oracle_step(ps, row_part, cm, z, V), V)


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("V,K,B,M", [
    (20008, 200, 1, 3), (20008, 200, 2, 2), (20008, 200, 3, 2), (20008, 2048, 2, 2), (20008, 2048, 3, 2), (20008, 2048, 13, 3),
    (30000, 3072, 3, 2), (30000, 3073, 3, 2), (30000, 8000, 4, 2), (128256, 300, 5, 5), (102400, 300, 3, 2), (102408, 300, 3, 2), (256000, 300, 2, 2),
    (40000, 1024, 26, 2), (40000, 1023, 40, 4)])
def test_several_masks_per_row(V, K, B, M, dtype):
    test_gpu_multi_mask.test_multi_mask_shapes(V, K, B, M, dtype)
