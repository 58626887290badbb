"""The one-launch step of a short batch (a thread-block cluster per row or few rows) against the CPU oracle, at the edges of its
shapes: rows per cluster, runs and chunks of the warps, tokens outside the vectors, rows off the vector grid, rows without a
partition, and the calls that have to stay with two launches."""
import numpy as np
import pytest
import torch

import synth
from synth import rng
from paper_2605_29986_b200 import binding as cz
from _gpu_util import Ctx, assert_close_log, compare_step, dev, oracle_step, run_fused
from test_gpu_sample import check_sample, run_sample

pytestmark = pytest.mark.gpu


def inputs(V, K, B, dtype, tag, p=0.2):
    part = synth.zipf_partition(V, K, seed=tag)
    cm = synth.class_mask_bernoulli(K, B, p, rng.stream_key(rng.SEED_BASE, 920, tag, V))
    cm[B // 2] = 0  # a row with nothing allowed
    return part, cm, synth.logits_normal(B, V, 2.0, dtype, (921, tag, V))


# V: less than an octet, one chunk per block and one token more or less, every warp a short run, eight chunks a warp;
# B: clusters of 1, 2, 3 and 4 rows, the last one not full
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("V,K,B", [(3, 2, 2), (8, 3, 9), (65, 33, 7), (4096, 64, 3), (4097, 65, 5), (65528, 2047, 16), (65544, 2048, 17), (128256, 2048, 31),
                                   (131072, 8192, 47), (100001, 5000, 63), (99999, 300, 33), (200008, 16384, 7)])
def test_greedy_and_sampling(V, K, B, dtype):
    part, cm, z = inputs(V, K, B, dtype, 1)
    want = oracle_step([part], None, cm, z, V, want_full=True)
    with Ctx([part]) as ctx:
        before = cz.cfgzip_launch_count(ctx.h)
        compare_step(run_fused(ctx, None, cm, z, V), want, V)
        compare_step(run_fused(ctx, None, cm, z, V, want_full=True, want_vm=False), want, V)
        if B <= 16:
            assert cz.cfgzip_launch_count(ctx.h) - before == 2  # two steps
        for u in (np.zeros(B), np.full(B, 1 - 2.0 ** -24), np.linspace(0, 0.99, B)):
            u = u.astype(np.float32)
            check_sample(run_sample(ctx, None, cm, z, V, u, 1.25), [part], None, cm, z, V, u, 1.25)
        assert cz.cfgzip_poll_status(ctx.h) == (5 * int((want["argmax"] < 0).sum()), 0, 0)  # five steps
        cz.cfgzip_set_tuning(ctx.h, "one_launch", 0)
        before = cz.cfgzip_launch_count(ctx.h)
        compare_step(run_fused(ctx, None, cm, z, V), want, V)
        assert cz.cfgzip_launch_count(ctx.h) - before >= 2


@pytest.mark.parametrize("V", [20000, 20003])
@pytest.mark.parametrize("B", [2, 20, 32])
def test_rows_of_several_partitions(V, B):
    parts = [synth.zipf_partition(V, k, seed=i) for i, k in enumerate((50, 333, 700))]
    row_part = (np.arange(B) * 7 % 3).astype(np.int32)
    cm = synth.class_mask_bernoulli(700, B, 0.2, rng.stream_key(rng.SEED_BASE, 922))
    z = synth.logits_normal(B, V, 2.0, "bf16", (923,))
    want = oracle_step(parts, row_part, cm, z, V)
    with Ctx(parts) as ctx:
        d_rp = torch.from_numpy(row_part).cuda()
        cz.cfgzip_plan_rows(ctx.h, ctx.ids[0], d_rp, B)
        compare_step(run_fused(ctx, row_part, cm, z, V), want, V)
        with pytest.raises(Exception):  # an explicit vector ends the kept grouping
            cz.cfgzip_map_tokens(ctx.h, ctx.ids[0], cz.ROWS_AS_PLANNED, d_rp, d_rp, B)
        bad = row_part.copy()
        bad[1] = 9
        got = run_fused(ctx, bad, cm, z, V)
        assert got["argmax"][1] == -7 and np.array_equal(got["logits"][1], z[1]) and cz.cfgzip_poll_status(ctx.h)[2] == 1
        keep = np.arange(B) != 1
        for key in ("argmax", "rep", "vocab_mask"):
            assert np.array_equal(got[key][keep], want[key][keep])


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
def test_ties_and_waits(dtype):
    # equal maxima in the head, in several blocks and in the tail: the lowest id wins; a wait reported as run out surfaces
    V, B = 30005, 12
    part, cm, z = inputs(V, 100, B, dtype, 3)
    cm[:] = 0xFFFFFFFF
    for b in range(B):
        z[b, [(b % 9), 5000 + b, 20000, V - 1 - (b % 7)]] = 50.0 if dtype == "f32" else 0x4248
    want = oracle_step([part], None, cm, z, V)
    with Ctx([part]) as ctx:
        compare_step(run_fused(ctx, None, cm, z, V), want, V)
        assert cz.cfgzip_poll_status(ctx.h) == (0, 0, 0)
        cz.cfgzip_set_tuning(ctx.h, "test_expire_waits", 1)
        run_fused(ctx, None, cm, z, V)
        assert cz.load_library().cfgzip_poll_status(ctx.h, None, None, None, None) == cz.E_CUDA
        cz.cfgzip_set_tuning(ctx.h, "test_expire_waits", 0)
        compare_step(run_fused(ctx, None, cm, z, V), want, V)


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("V", [20000, 20003])
def test_no_weight_is_no_draw(V, dtype):
    # values outside the contract: a row without a weight to draw by says so, as it does in two launches, and keeps no earlier token
    B = 9
    part, cm, z = inputs(V, 100, B, dtype, 4)
    cm[:] = 0xFFFFFFFF
    bad = (1, 4, 8)
    for b, t in zip(bad, (0, 777, V - 1)):
        z[b, t] = np.inf if dtype == "f32" else 0x7F80
    z[4, :] = z[4, 777]
    u = np.linspace(0, 0.99, B).astype(np.float32)
    ok = [b for b in range(B) if b not in bad]
    with Ctx([part]) as ctx:
        for one_launch in (1, 0):
            cz.cfgzip_set_tuning(ctx.h, "one_launch", one_launch)
            before = cz.cfgzip_launch_count(ctx.h)
            got = run_sample(ctx, None, cm, z, V, u, 1.0)
            assert cz.cfgzip_launch_count(ctx.h) - before == 2 - one_launch
            for b in bad:
                assert got["token"][b] == -1 and got["rep"][b] == -1 and np.isneginf(got["lse"][b]) and np.isneginf(got["logp_token"][b])
            check_sample({k: v[ok] for k, v in got.items()}, [part], None, cm[ok], z[ok], V, u[ok], 1.0)


def test_a_refused_knob_changes_nothing():
    V, B = 20000, 9
    part, cm, z = inputs(V, 100, B, "bf16", 5)
    lib = cz.load_library()

    def launches(ctx):
        before = cz.cfgzip_launch_count(ctx.h)
        run_fused(ctx, None, cm, z, V)
        return cz.cfgzip_launch_count(ctx.h) - before

    with Ctx([part]) as ctx:
        for knob, value in ((b"ctas_per_sm", 0), (b"row_warps", 3), (b"token_warps", 17), (b"pipe_warps", 0), (b"waves", 0), (b"fold", 3),
                            (b"lane_octets", 3), (b"pipe_depth", 1), (b"nonsense", 1)):
            assert lib.cfgzip_set_tuning(ctx.h, knob, value) == cz.E_ARG and launches(ctx) == 1, knob
        assert lib.cfgzip_set_tuning(ctx.h, b"row_warps", 1) == 0 and launches(ctx) == 2


def limit_rows(V, dtype):
    """Rows whose sums are at the ends of their range: every value close to the one below which a logit weighs nothing, fill values beside one or
    many others, fill values first, and a climb of 400 nats that moves the sums' reference again and again."""
    part, cm, z = inputs(V, 50, 6, "f32", 6)
    cm[:] = 0xFFFFFFFF
    t = np.arange(V, dtype=np.float32)
    z[0] = -1.2e9 - 1e4 * t
    z[0, 5] = -1e9  # (one largest value, also when rounded to bf16: the log of a tie is lost beside 1e9)
    z[1] = -1e30
    z[1, V // 3] = 0.0
    z[2, ::2] = -3e38
    z[3, 4096:12288] = -1e10
    z[4] = -200.0 + 400.0 * t / V
    z[5, :8000] = -1e37
    return part, cm, rng.f32_to_bf16_bits(z.reshape(-1)).reshape(z.shape) if dtype == "bf16" else z


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("V", [20000, 20003])
@pytest.mark.parametrize("one_launch", [1, 0])
def test_sums_at_the_ends_of_their_range(V, dtype, one_launch):
    part, cm, z = limit_rows(V, dtype)
    B = len(z)
    u = np.linspace(0, 0.99, B).astype(np.float32)
    with Ctx([part]) as ctx:
        cz.cfgzip_set_tuning(ctx.h, "one_launch", one_launch)
        compare_step(run_fused(ctx, None, cm, z, V), oracle_step([part], None, cm, z, V), V)
        check_sample(run_sample(ctx, None, cm, z, V, u, 1.0), [part], None, cm, z, V, u, 1.0)
        # very low temperatures: logits whose z / T stays where 1e-4 can be told, then ordinary ones, of which the largest is drawn
        for inv_t, sigma in ((200.0, 0.02), (1e6, 4e-6)):
            y = synth.logits_normal(B, V, sigma, dtype, (924, V))
            check_sample(run_sample(ctx, None, cm, y, V, u, inv_t), [part], None, cm, y, V, u, inv_t)
        y = synth.logits_normal(B, V, 2.0, "f32", (925, V))
        y[np.arange(B), 1000 * np.arange(B) + 3] = 16.0
        got = run_sample(ctx, None, cm, y, V, u, 1e6)
        assert np.array_equal(got["token"], 1000 * np.arange(B) + 3) and np.all(got["lse"] == 16e6) and np.all(got["logp_token"] == 0)


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("kind,V,B", [("one launch", 20000, 20), ("streaming", 40000, 96), ("streaming", 40003, 96), ("registers", 20000, 40),
                                      ("class lists", 20000, 20), ("few tokens", 60000, 96), ("several masks", 20000, 3)])
def test_fill_values_weigh_nothing(kind, V, B, dtype):
    # allowed tokens that the program in front has set to a large negative number, whole runs of them
    K = 60
    part = synth.zipf_partition(V, K, seed=9)
    M = 5 if kind == "several masks" else 1
    cm = synth.class_mask_bernoulli(K, B * M, 0.1 if kind in ("class lists", "few tokens") else 0.7, rng.stream_key(rng.SEED_BASE, 926, V))
    cm[:, 0] |= 1
    z = synth.logits_normal(B, V, 2.0, "f32", (927, V))
    for b in range(B):
        z[b, 300 * b : 300 * b + V // 2] = (-1e9, -1e10, -1e30, -1e37, -3e38)[b % 5]
    if dtype == "bf16":
        z = rng.f32_to_bf16_bits(z.reshape(-1)).reshape(z.shape)
    many = np.repeat(z, M, axis=0)
    want = oracle_step([part], None, cm, many, V)
    with Ctx([part]) as ctx:
        if kind != "one launch":
            cz.cfgzip_set_tuning(ctx.h, "one_launch", 0)
        if kind == "registers":
            cz.cfgzip_set_tuning(ctx.h, "pipeline", 0)
        if M > 1:
            d_z, d_cm = dev(z), dev(cm)
            tok, rep = (torch.zeros(B * M, dtype=torch.int32, device="cuda") for _ in range(2))
            lp, lse = (torch.zeros(B * M, device="cuda") for _ in range(2))
            cz.cfgzip_multi_mask_logsoftmax_argmax(ctx.h, ctx.ids[0], d_cm, cm.shape[1], M, d_z, cz.BF16 if dtype == "bf16" else cz.F32, V, B,
                                                   None, 0, tok, rep, lp, lse)
            assert np.array_equal(tok.cpu().numpy(), want["argmax"]) and np.array_equal(rep.cpu().numpy(), want["rep"])
            assert_close_log(lse.cpu().numpy(), want["lse"], "lse")
            return
        compare_step(run_fused(ctx, None, cm, z, V, mode=cz.SPARSE if kind in ("class lists", "few tokens") else cz.DENSE), want, V)
        if kind in ("one launch", "streaming"):
            u = rng.uniform(rng.stream_key(928, V), B).astype(np.float32)
            check_sample(run_sample(ctx, None, cm, z, V, u, 1.3), [part], None, cm, z, V, u, 1.3)
