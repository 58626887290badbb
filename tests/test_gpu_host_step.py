"""cfgzip_decode_step_host: what it counts and what it leaves alone is the same with pinned and with pageable buffers."""
import numpy as np
import pytest
import torch

import synth
from synth import rng
from paper_2605_29986_b200 import binding as cz
from _gpu_util import Ctx, dtype_code

pytestmark = pytest.mark.gpu


def buffers(B, V, z, pinned):
    made = [torch.from_numpy(np.full_like(z, 7).view(np.int16 if z.dtype == np.uint16 else np.float32)),
            torch.full((B, (V + 31) // 32), 0x5A5A5A5A, dtype=torch.int32)]
    made += [torch.full((B,), -7, dtype=torch.int32) for _ in range(2)] + [torch.full((B,), 123.0) for _ in range(2)]
    return [t.pin_memory() for t in made] if pinned else made


def pin(a, pinned):
    t = torch.from_numpy(a.view(np.int16 if a.dtype == np.uint16 else np.int32 if a.dtype == np.uint32 else a.dtype))
    return t.pin_memory() if pinned else t


@pytest.mark.parametrize("pinned", [False, True])
@pytest.mark.parametrize("V,B,dtype", [(3000, 5, "f32"), (9001, 70, "bf16")])
def test_rows_without_a_partition_are_counted_once(V, B, dtype, pinned):
    ps = [synth.zipf_partition(V, 100, seed=90 + i) for i in range(2)]
    row_part = (np.arange(B) % 2).astype(np.int32)
    row_part[1::4] = 9
    cm = synth.class_mask_bernoulli(100, B, 0.3, rng.stream_key(rng.SEED_BASE, 920, V))
    z = synth.logits_normal(B, V, 2.0, dtype, (921, V))
    with Ctx(ps) as ctx:
        masked, vm, am, rep, lse, lpa = buffers(B, V, z, pinned)
        cz.cfgzip_decode_step_host(ctx.h, ctx.ids[0], row_part, pin(cm, pinned), cm.shape[1], pin(z, pinned), dtype_code(z), B, None, vm, am, rep,
                                   lpa, lse, cz.DENSE)
        assert cz.cfgzip_poll_status(ctx.h) == (0, 0, len(row_part[1::4]))


@pytest.mark.parametrize("want_masked", [False, True])
@pytest.mark.parametrize("pinned", [False, True])
@pytest.mark.parametrize("V,B,dtype", [(3000, 5, "f32"), (9001, 70, "bf16")])
def test_rows_without_a_partition_are_left_alone(V, B, dtype, pinned, want_masked):
    # a first call with every row leaves its results in the context's staging memory: none of them may come out of the second
    ps = [synth.zipf_partition(V, 100, seed=90 + i) for i in range(2)]
    cm = synth.class_mask_bernoulli(100, B, 0.3, rng.stream_key(rng.SEED_BASE, 922, V))
    z = synth.logits_normal(B, V, 2.0, dtype, (923, V))
    row_part = (np.arange(B) % 2).astype(np.int32)
    with Ctx(ps) as ctx:
        def call(parts):
            masked, vm, am, rep, lse, lpa = buffers(B, V, z, pinned)
            cz.cfgzip_decode_step_host(ctx.h, ctx.ids[0], parts, pin(cm, pinned), cm.shape[1], pin(z, pinned), dtype_code(z), B,
                                       masked if want_masked else None, vm, am, rep, lpa, lse, cz.DENSE)
            return [t.numpy().copy() for t in (masked, vm, am, rep, lse, lpa)]

        want, untouched = call(row_part), [t.numpy() for t in buffers(B, V, z, False)]
        some = row_part.copy()
        some[[0, 2, B - 1]] = (9, -1, 2)
        left = np.isin(np.arange(B), [0, 2, B - 1])
        for got, full, before in zip(call(some), want, untouched):
            assert np.array_equal(got[left], before[left])
            assert np.array_equal(got[~left], full[~left]) or np.abs(got[~left] - full[~left]).max() <= 1e-5  # (other row groups: other sums)
