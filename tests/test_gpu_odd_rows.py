"""Rows that do not start on a vector boundary (an odd vocabulary packed end to end, a view into a larger buffer): the
streaming kernel's shifted variant and the sampling kernels behind it, against the CPU oracle."""
import numpy as np
import pytest
import torch

import synth
from synth import rng
from paper_2605_29986_b200 import binding as cz
from _gpu_util import Ctx, compare_step, dev, dtype_code, host, oracle_step, run_fused
from test_gpu_sample import check_sample, run_sample
from test_gpu_sample_filtered import check_filtered, run_filtered

pytestmark = pytest.mark.gpu


def inputs(V, K, B, dtype, tag, stride=None, p=0.3, sigma=2.0):
    part = synth.zipf_partition(V, K, seed=tag)
    cm = synth.class_mask_bernoulli(K, B, p, rng.stream_key(rng.SEED_BASE, 901, tag, V))
    z = synth.logits_normal(B, stride or V, sigma, dtype, (902, tag, V))
    return part, cm, z


# one octet and less, the edges of a chunk of 31 vectors, tails of every length, rows enough for several groups
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("V,B", [(1, 3), (7, 9), (9, 8), (17, 33), (247, 8), (249, 40), (255, 17), (257, 31), (505, 8),
                                 (10001, 70), (20002, 1), (20003, 5), (20005, 32), (20007, 65), (70009, 33)])
def test_greedy(V, B, dtype):
    K = max(1, min(300, V // 2))
    part, cm, z = inputs(V, K, B, dtype, 1)
    with Ctx([part]) as ctx:
        compare_step(run_fused(ctx, None, cm, z, V), oracle_step([part], None, cm, z, V), V, "V=%d B=%d" % (V, B))


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("offset", [1, 3, 6, 7])
def test_view_into_a_buffer(offset, dtype):
    V, K, B, stride = 3001, 90, 11, 3010
    part, cm, z = inputs(V, K, B, dtype, 2, stride)
    want = oracle_step([part], None, cm, z, V)
    flat = np.zeros(offset + B * stride + 8, dtype=z.dtype)
    flat[offset:offset + B * stride] = z.reshape(-1)
    with Ctx([part]) as ctx:
        d, d_cm, es = dev(flat), dev(cm), z.dtype.itemsize
        VW = (V + 31) // 32
        d_vm, d_am = torch.zeros((B, VW), dtype=torch.int32, device="cuda"), torch.zeros(B, dtype=torch.int32, device="cuda")
        d_rep, d_lse, d_lpa = torch.zeros_like(d_am), torch.zeros(B, device="cuda"), torch.zeros(B, device="cuda")
        cz.cfgzip_masked_logsoftmax_argmax(ctx.h, ctx.ids[0], None, d_cm, cm.shape[1], d.data_ptr() + offset * es, dtype_code(z),
                                           stride, B, d_vm, VW, d_am, d_rep, d_lpa, d_lse)
        torch.cuda.synchronize()
        back = host(d, z.dtype)
        rows = back[offset:offset + B * stride].reshape(B, stride)
        compare_step(dict(logits=rows, vocab_mask=host(d_vm, np.uint32), argmax=d_am.cpu().numpy(), rep=d_rep.cpu().numpy(),
                          lse=d_lse.cpu().numpy(), logp_argmax=d_lpa.cpu().numpy()), want, V)
        assert np.array_equal(rows[:, V:], z[:, V:]) and not back[:offset].any() and not back[offset + B * stride:].any()


def test_ties_and_maxima_at_the_edges():
    V, K, B = 2005, 40, 16
    part, cm, z = inputs(V, K, B, "f32", 3)
    cm[:] = 0xFFFFFFFF
    for b in range(B):  # equal maxima in front of, inside and behind the vectors of the row
        z[b, [(b % 9), 8 * b + 5, V - 1 - (b % 7)]] = 50.0
    with Ctx([part]) as ctx:
        compare_step(run_fused(ctx, None, cm, z, V), oracle_step([part], None, cm, z, V), V)


def test_mixed_partitions():
    V, B = 9001, 77
    parts = [synth.zipf_partition(V, k, seed=i) for i, k in enumerate((50, 333, 700))]
    row_part = (np.arange(B) * 7 % 3).astype(np.int32)
    cm = synth.class_mask_bernoulli(700, B, 0.2, rng.stream_key(rng.SEED_BASE, 903))
    z = synth.logits_normal(B, V, 2.0, "bf16", (904,))
    with Ctx(parts) as ctx:
        compare_step(run_fused(ctx, row_part, cm, z, V), oracle_step(parts, row_part, cm, z, V), V)


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("V,B", [(7, 4), (249, 9), (5003, 33), (40001, 40)])
def test_sampling(V, B, dtype):
    part, cm, z = inputs(V, max(1, min(200, V // 3)), B, dtype, 5)
    for n, fill in enumerate((0.0, 0.37, 0.999999)):
        u = np.full(B, fill, dtype=np.float32) if n != 1 else np.linspace(0, 0.99, B, dtype=np.float32)
        with Ctx([part]) as ctx:
            got = run_sample(ctx, None, cm, z, V, u, 1.25)
            check_sample(got, [part], None, cm, z, V, u, 1.25, "V=%d" % V)


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("V,B,inv_t,top_k,top_p", [(7, 4, 1.0, 3, 0.9), (249, 9, 5.0, 20, 1.0), (5003, 33, 1.0, 0, 0.9),
                                                   (40001, 40, 1.0, 0, 0.95), (40001, 80, 5.0, 50, 0.9)])
def test_filtered_sampling(V, B, inv_t, top_k, top_p, dtype):
    part, cm, z = inputs(V, max(1, min(200, V // 3)), B, dtype, 6)
    u = np.linspace(0, 0.99, B, dtype=np.float32)
    with Ctx([part]) as ctx:
        got = run_filtered(ctx, None, cm, z, V, u, inv_t, top_k, top_p)
        check_filtered(got, [part], None, cm, z, V, u, inv_t, top_k, top_p, "V=%d" % V)


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("V,B", [(9001, 5), (28864, 150)])
def test_filtered_cut_below_a_peak(V, B, dtype):
    # a few large logits hold most of the weight and the nucleus ends in the thin top of the bulk below them, row by row a
    # little further down: the steps around the cut hold few tokens, those below it thousands
    K = 200
    part, cm, z = inputs(V, K, B, dtype, 430, p=0.9, sigma=1.0)
    f = z if dtype == "f32" else (z.astype(np.uint32) << 16).view(np.float32)
    f = f.copy()
    f[:, 11 : 11 + 6] = np.linspace(4.0, 9.0, B, dtype=np.float32)[:, None] + np.arange(6, dtype=np.float32) / 8
    z = f if dtype == "f32" else (f.view(np.uint32) >> 16).astype(np.uint16)
    u = rng.uniform(rng.stream_key(431, B), B).astype(np.float32)
    with Ctx([part]) as ctx:
        for top_p in (0.5, 0.9):
            got = run_filtered(ctx, None, cm, z, V, u, 1.0, 0, top_p)
            close, near = check_filtered(got, [part], None, cm, z, V, u, 1.0, 0, top_p, "p=%g" % top_p)
            assert near <= 1


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("V,B,p,step", [(20000, 150, 0.9, 1 / 16), (20001, 9, 0.9, 1 / 4), (9001, 40, 0.01, 0.0), (57592, 160, 0.01, 0.0)])
def test_filtered_top_p_alone(V, B, p, step, dtype):
    # logits on a grid: hundreds of tokens per value, so that the first window holds one of them and the cut may lie in the next;
    # few allowed tokens: hardly more than one to a run of the row, the run maxima fall short of the weight the nucleus needs
    part, cm, z = inputs(V, 300, B, dtype, 432, p=p)
    if step:
        f = z if dtype == "f32" else (z.astype(np.uint32) << 16).view(np.float32)
        f = np.round(f / step).astype(np.float32) * np.float32(step)
        z = f if dtype == "f32" else (f.view(np.uint32) >> 16).astype(np.uint16)
    u = rng.uniform(rng.stream_key(433, B), B).astype(np.float32)
    with Ctx([part]) as ctx:
        for inv_t, top_p in ((1.0, 0.5), (1.0, 0.9), (1.4, 0.95), (5.0, 0.9)):
            got = run_filtered(ctx, None, cm, z, V, u, inv_t, 0, top_p)
            close, near = check_filtered(got, [part], None, cm, z, V, u, inv_t, 0, top_p, "1/T=%g p=%g" % (inv_t, top_p))
            assert near <= 1


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("V,pad,B,parts", [(7, 1, 64, 1), (15, 1, 70, 1), (16, 0, 64, 1), (31, 1, 65, 1), (264, 0, 64, 1), (513, 7, 97, 1),
                                           (8200, 0, 100, 3), (30000, 0, 64, 1), (70007, 1, 129, 2)])
def test_rows_that_allow_few_tokens(V, pad, B, parts, dtype):
    """Vectors of 32 bytes (odd octets left over, rows on a 16-byte but not on a 32-byte grid), queues that never fill and that
    overflow at once (some rows allow everything, some nothing)."""
    pad = (-(V + pad)) % 8 + pad
    K = max(1, min(128, V // 4))
    ps = [synth.zipf_partition(V, K, seed=40 + i) for i in range(parts)]
    row_part = None if parts == 1 else (np.arange(B) * 5 % parts).astype(np.int32)
    cm = synth.class_mask_bernoulli(K, B, 0.03, rng.stream_key(rng.SEED_BASE, 905, V))
    cm[3], cm[B - 1], cm[B // 2] = 0xFFFFFFFF, 0xFFFFFFFF, 0
    z = synth.logits_normal(B, V + pad, 2.0, dtype, (906, V))
    with Ctx(ps) as ctx:
        got = run_fused(ctx, row_part, cm, z, V, stride=V + pad, mode=cz.SPARSE)
        compare_step(got, oracle_step(ps, row_part, cm, z, V), V)
        assert np.array_equal(got["logits"][:, V:].view(np.uint8), z[:, V:].view(np.uint8))


@pytest.mark.parametrize("pad", [0, 1])
@pytest.mark.parametrize("V,counts", [(9000, (33, 1, 64, 2)), (70008, (97, 0, 3, 8)), (20000, (5, 1, 1, 1)), (1000, (31, 33, 40, 200))])
def test_groups_of_very_different_size(V, counts, pad):
    """The blocks of a mixed batch are shared out by the sizes of its row groups: greedy (folded in the kernel too), sampling,
    filtered sampling."""
    parts = [synth.zipf_partition(V, k, seed=60 + i) for i, k in enumerate((50, 333, 700, 64))]
    row_part = np.random.RandomState(V).permutation(np.repeat(np.arange(4), counts)).astype(np.int32)
    B, stride = len(row_part), V + 8 * (1 - pad) + pad
    cm = synth.class_mask_bernoulli(700, B, 0.2, rng.stream_key(rng.SEED_BASE, 907, V))
    cm[:, 0] |= 1
    z = synth.logits_normal(B, stride, 2.0, "bf16", (908, V))
    u = np.linspace(0, 0.99, B, dtype=np.float32)
    want = oracle_step(parts, row_part, cm, z, V)
    with Ctx(parts) as ctx:
        for fold in (0, 1, 2):
            cz.cfgzip_set_tuning(ctx.h, "fold", fold)
            compare_step(run_fused(ctx, row_part, cm, z, V, stride=stride), want, V, "fold %d" % fold)
        cz.cfgzip_set_tuning(ctx.h, "fold", 0)
        check_sample(run_sample(ctx, row_part, cm, z, V, u, 1.5, stride=stride), parts, row_part, cm, z, V, u, 1.5)
        check_filtered(run_filtered(ctx, row_part, cm, z, V, u, 1.5, 30, 0.9, stride=stride), parts, row_part, cm, z, V, u, 1.5, 30, 0.9)


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("V,B,parts,p", [(1001, 1, 1, 0.3), (25000, 8, 1, 0.3), (25003, 9, 2, 0.3), (9000, 70, 1, 0.002), (9000, 130, 3, 0.2)])
def test_host_step_with_pinned_buffers(V, B, parts, p, dtype):
    """Copies in, expansion, step and copies out on streams of their own: one row chunk, several, a short last one."""
    ps = [synth.zipf_partition(V, 300, seed=70 + i) for i in range(parts)]
    row_part = None if parts == 1 else (np.arange(B) * 3 % parts).astype(np.int32)
    cm = synth.class_mask_bernoulli(300, B, p, rng.stream_key(rng.SEED_BASE, 909, V))
    VW = (V + 31) // 32

    def pin(a):
        return torch.from_numpy(a.view(np.int16 if a.dtype == np.uint16 else np.int32 if a.dtype == np.uint32 else a.dtype)).pin_memory()

    with Ctx(ps) as ctx:
        for step in range(2):
            z = synth.logits_normal(B, V, 2.0, dtype, (910, V, step))
            want = oracle_step(ps, row_part, cm, z, V)
            for want_masked in (False, True):
                d_z, d_cm, vm = pin(z), pin(cm), torch.zeros((B, VW), dtype=torch.int32).pin_memory()
                masked = torch.zeros_like(d_z).pin_memory() if want_masked else None
                am, rep = np.full(B, -7, dtype=np.int32), np.full(B, -7, dtype=np.int32)
                lse, lpa = np.full(B, 9, dtype=np.float32), np.full(B, 9, dtype=np.float32)
                cz.cfgzip_decode_step_host(ctx.h, ctx.ids[0], row_part, d_cm, cm.shape[1], d_z, dtype_code(z), B, masked, vm, am,
                                           rep, lpa, lse)
                assert np.array_equal(d_z.numpy().view(np.uint8), z.view(np.uint8))
                compare_step(dict(logits=masked.numpy().view(z.dtype) if want_masked else want["logits"],
                                  vocab_mask=vm.numpy().view(np.uint32), argmax=am, rep=rep, lse=lse, logp_argmax=lpa), want, V)
