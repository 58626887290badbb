"""Calls on either side of the lines at which a step takes another kernel, against the CPU oracle: rows that allow few tokens
(row count, classes, row length, mixed batches)."""
import numpy as np
import pytest

import synth
from synth import rng
from paper_2605_29986_b200 import binding as cz
from _gpu_util import Ctx, compare_step, oracle_step, run_fused

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("V,K,B,parts", [
    (9000, 300, 63, 1), (9000, 300, 64, 1),
    (60000, 4800, 64, 1), (60000, 5100, 64, 1), (60000, 16000, 64, 1),       # masks staged or not; two blocks per SM
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
