"""Class masks of every alignment against the CPU oracle: rows on 16-byte boundaries, row groups that are one piece of memory (its last
words by plain loads), and masks off every boundary, whole or a slice of 128 words at a time, in the streaming kernel, the kernel for
rows that allow few tokens, the expansion, several masks per row and mixed batches."""
import numpy as np
import pytest
import torch

import oracle
import synth
from synth import rng
from paper_2605_29986_b200 import binding as cz
from _gpu_util import Ctx, compare_step, dev, oracle_step

pytestmark = pytest.mark.gpu


def step(ctx, row_part, d_cm, stride, z, V, mode, masks_per_row=0):
    B = z.shape[0]
    rows = B * max(masks_per_row, 1)
    d_z = dev(z)
    d_vm = torch.zeros((rows, (V + 31) // 32), dtype=torch.int32, device="cuda")
    tok, rep = (torch.zeros(rows, dtype=torch.int32, device="cuda") for _ in range(2))
    lp, lse = (torch.zeros(rows, dtype=torch.float32, device="cuda") for _ in range(2))
    d_rp = None if row_part is None else dev(row_part)
    if masks_per_row:
        cz.cfgzip_multi_mask_logsoftmax_argmax(ctx.h, ctx.ids[0], d_cm, stride, masks_per_row, d_z, cz.BF16, z.shape[1], B, d_vm,
                                               d_vm.shape[1], tok, rep, lp, lse)
    else:
        cz.cfgzip_masked_logsoftmax_argmax(ctx.h, ctx.ids[0], d_rp, d_cm, stride, d_z, cz.BF16, z.shape[1], B, d_vm, d_vm.shape[1], tok,
                                           rep, lp, lse, None, mode)
    torch.cuda.synchronize()
    return {"vocab_mask": d_vm.cpu().numpy().view(np.uint32), "logits": d_z.cpu().numpy().view(np.uint16), "argmax": tok.cpu().numpy(), "rep": rep.cpu().numpy(),
            "logp_argmax": lp.cpu().numpy(), "lse": lse.cpu().numpy()}


def masks_on(cm, pad, offset):
    """The masks on the device, `pad` words between rows, `offset` words off a 16-byte boundary; nothing behind the last row's words."""
    B, KW = cm.shape
    n = offset + (B - 1) * (KW + pad) + KW
    flat = np.full(n + pad, 0xFFFFFFFF, dtype=np.uint32)
    for b in range(B):
        flat[offset + b * (KW + pad): offset + b * (KW + pad) + KW] = cm[b]
    return torch.from_numpy(flat[:n].view(np.int32)).cuda()[offset:]


@pytest.mark.parametrize("K,B", [(20, 65), (33, 33), (96, 97), (1500, 100), (2080, 64), (4100, 47), (8190, 34), (16420, 40), (20001, 66)])
@pytest.mark.parametrize("pad,offset", [(0, 0), (1, 0), (2, 0), (0, 1), (3, 2)])
def test_every_alignment(K, B, pad, offset):
    V = max(24000, K + 1000)
    part = synth.zipf_partition(V, K, seed=K)
    cm = synth.class_mask_bernoulli(K, B, 0.2, rng.stream_key(rng.SEED_BASE, 950, K))
    z = synth.logits_normal(B, V, 2.0, "bf16", (951, K))
    want = oracle_step([part], None, cm, z, V)
    with Ctx([part]) as ctx:
        cz.cfgzip_set_tuning(ctx.h, "one_launch", 0)
        d_cm = masks_on(cm, pad, offset)
        for mode in (cz.DENSE, cz.SPARSE):
            compare_step(step(ctx, None, d_cm, cm.shape[1] + pad, z, V, mode), want, V)


# A block of one or two warps, whose lanes take more than one piece each of a group's masks (20001 classes: 80128 bytes)
@pytest.mark.parametrize("knob,value", [("token_warps", 1), ("row_warps", 1), ("row_warps", 2), ("pipe_warps", 1)])
@pytest.mark.parametrize("K,V,B", [(16400, 24000, 448), (20001, 24000, 32)])
def test_few_warps_fetch_a_whole_block_of_masks(K, V, B, knob, value):
    part = synth.zipf_partition(V, K, seed=K)
    cm = synth.class_mask_bernoulli(K, B, 0.2, rng.stream_key(rng.SEED_BASE, 954, K))
    z = synth.logits_normal(B, V, 2.0, "bf16", (955, K))
    with Ctx([part]) as ctx:
        cz.cfgzip_set_tuning(ctx.h, knob, value)
        compare_step(step(ctx, None, masks_on(cm, 0, 0), cm.shape[1], z, V, cz.DENSE), oracle_step([part], None, cm, z, V), V)
        assert cz.cfgzip_poll_status(ctx.h) == (0, 0, 0)


@pytest.mark.parametrize("K", [50, 1500, 5000, 16420])
@pytest.mark.parametrize("pad,offset", [(0, 0), (3, 1)])
def test_several_masks_and_several_partitions(K, pad, offset):
    V, B, M = 24000, 5, 9
    parts = [synth.zipf_partition(V, k, seed=k) for k in (K, K // 2)]
    cm = synth.class_mask_bernoulli(K, B * M, 0.2, rng.stream_key(rng.SEED_BASE, 952, K))
    z = synth.logits_normal(B, V, 2.0, "bf16", (953, K))
    many = np.repeat(z, M, axis=0)
    want = oracle_step(parts[:1], None, cm, many, V)
    d_cm = masks_on(cm, pad, offset)
    with Ctx(parts) as ctx:
        got = step(ctx, None, d_cm, cm.shape[1] + pad, z, V, cz.DENSE, masks_per_row=M)
        for key in ("vocab_mask", "argmax", "rep"):
            assert np.array_equal(got[key], want[key]), key
        assert np.allclose(got["lse"], want["lse"], rtol=0, atol=1e-4)  # as everywhere: f32 sums against f64
        row_part = (np.arange(B * M) % 2).astype(np.int32)
        compare_step(step(ctx, row_part, d_cm, cm.shape[1] + pad, many, V, cz.DENSE), oracle_step(parts, row_part, cm, many, V), V)


# Class tables that leave no room for a slice of the masks beside them, and one word of masks more than fits: several masks per row as far as
# the table goes (57536 classes), one mask per row beyond
@pytest.mark.parametrize("K", [46500, 48300, 53000, 53600, 57000, 57536, 57537])
@pytest.mark.parametrize("pad,offset", [(0, 0), (1, 0), (0, 1)])
def test_tables_that_fill_shared_memory(K, pad, offset):
    V, B, M = 60032, 3, 3
    part = synth.zipf_partition(V, K, seed=K)
    cm = synth.class_mask_bernoulli(K, B * M, 0.2, rng.stream_key(rng.SEED_BASE, 956, K))
    z = synth.logits_normal(B, V, 2.0, "bf16", (957, K))
    many = np.repeat(z, M, axis=0)
    want = oracle_step([part], None, cm, many, V)
    d_cm = masks_on(cm, pad, offset)
    with Ctx([part]) as ctx:
        cz.cfgzip_set_tuning(ctx.h, "one_launch", 0)
        compare_step(step(ctx, None, d_cm, cm.shape[1] + pad, many, V, cz.DENSE), want, V)
        if K > 57536:
            with pytest.raises(cz.CfgzipError):
                step(ctx, None, d_cm, cm.shape[1] + pad, z, V, cz.DENSE, masks_per_row=M)
            return
        got = step(ctx, None, d_cm, cm.shape[1] + pad, z, V, cz.DENSE, masks_per_row=M)
        for key in ("vocab_mask", "argmax", "rep"):
            assert np.array_equal(got[key], want[key]), key
        assert np.allclose(got["lse"], want["lse"], rtol=0, atol=1e-4)  # as everywhere: f32 sums against f64
