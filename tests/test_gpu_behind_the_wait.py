"""Batches of many and of few row groups by turns, with programmatic launches: every kernel of a call reads the row plan (and what else
the kernel in front of it has just written) behind its wait, so that no group of the call before is taken for one of this call."""
import numpy as np
import pytest
import torch

import synth
from synth import rng
from paper_2605_29986_b200 import binding as cz
from _gpu_util import Ctx, compare_step, dev, oracle_step
from test_gpu_sample import check_sample
from test_gpu_sample_filtered import check_filtered

pytestmark = pytest.mark.gpu

V, K, B, TURNS = 20000, 300, 96, 200


class Batch:
    """Rows of some partitions, with results of their own for every kind of call."""

    def __init__(self, parts, n_used, tag):
        self.row_part = (rng.uniform(rng.stream_key(960, tag), B) * n_used).astype(np.int32)
        self.cm = synth.class_mask_n_classes(K, B, 1, 5, rng.stream_key(961, tag))
        self.z = synth.logits_normal(B, V, 2.0, "bf16", (962, tag))
        self.u = rng.uniform(rng.stream_key(963, tag), B).astype(np.float32)
        self.want = oracle_step(parts, self.row_part, self.cm, self.z, V)
        self.d_rp, self.d_cm, self.d_u = dev(self.row_part), dev(self.cm), dev(self.u)
        self.host = [torch.from_numpy(a).pin_memory() for a in (self.cm.view(np.int32), self.z.view(np.int16))]
        self.out = {}

    def buffers(self, kind):
        if kind not in self.out:
            where = dict(pin_memory=True) if kind == "host" else dict(device="cuda")
            made = [torch.empty((B, (V + 31) // 32), dtype=torch.int32, **where)] + [torch.empty(B, dtype=torch.int32, **where) for _ in range(2)]
            made += [torch.empty(B, dtype=torch.float32, **where) for _ in range(2)]
            self.out[kind] = (dev(self.z), made)
        return self.out[kind]

    def call(self, ctx, kind):
        z, (vm, tok, rep, logp, lse) = self.buffers(kind)
        vm.fill_(0x5A5A5A5A)
        tok.fill_(-7)
        rep.fill_(-7)
        h, part, KW, VW = ctx.h, ctx.ids[0], self.cm.shape[1], vm.shape[1]
        if kind in ("step", "few"):
            full = torch.empty((B, V), device="cuda") if kind == "step" else None
            cz.cfgzip_masked_logsoftmax_argmax(h, part, self.d_rp, self.d_cm, KW, z, cz.BF16, V, B, vm, VW, tok, rep, logp, lse, full,
                                               cz.DENSE if kind == "step" else cz.SPARSE)
            return full
        if kind == "sample":
            cz.cfgzip_masked_sample(h, part, self.d_rp, self.d_cm, KW, z, cz.BF16, V, B, vm, VW, self.d_u, 1.0, tok, rep, logp, lse, cz.DENSE)
        elif kind == "filtered":
            cz.cfgzip_masked_sample_filtered(h, part, self.d_rp, self.d_cm, KW, z, cz.BF16, V, B, vm, VW, self.d_u, 1.0, 20, 0.9, tok, rep,
                                             logp, lse, cz.DENSE)
        elif kind == "expand":
            cz.cfgzip_expand_mask(h, part, self.d_rp, self.d_cm, KW, vm, VW, B, cz.DENSE)
            cz.cfgzip_mask_logits(h, z, cz.BF16, V, B, V, vm, VW)
        else:
            cz.cfgzip_decode_step_host(h, part, self.row_part, self.host[0], KW, self.host[1], cz.BF16, B, None, vm, tok, rep, logp, lse, cz.DENSE)

    def results(self, kind):
        z, (vm, tok, rep, logp, lse) = self.buffers(kind)
        return dict(logits=z.cpu().numpy().view(np.uint16), vocab_mask=vm.cpu().numpy().view(np.uint32), argmax=tok.cpu().numpy(),
                    token=tok.cpu().numpy(), rep=rep.cpu().numpy(), lse=lse.cpu().numpy(), logp_argmax=logp.cpu().numpy(),
                    logp_token=logp.cpu().numpy())


@pytest.mark.parametrize("kind", ["step", "few", "sample", "filtered", "expand", "host"])
def test_batches_of_many_and_few_groups_by_turns(kind):
    parts = [synth.zipf_partition(V, K, seed=i) for i in range(8)]
    batches = [Batch(parts, n, n) for n in (8, 1, 3)]
    with Ctx(parts) as ctx:
        cz.cfgzip_set_tuning(ctx.h, "pdl", 2)
        kept = []
        for turn in range(TURNS):
            full = [b.call(ctx, kind) for b in batches]
            now = [b.buffers(kind)[1][:3] + [f] for b, f in zip(batches, full)]
            if turn == 0:
                torch.cuda.synchronize()
                for b in batches:
                    got = b.results(kind)
                    if kind == "sample":
                        check_sample(got, parts, b.row_part, b.cm, b.z, V, b.u, 1.0)
                    elif kind == "filtered":
                        check_filtered(got, parts, b.row_part, b.cm, b.z, V, b.u, 1.0, 20, 0.9)
                    elif kind == "expand":
                        assert np.array_equal(got["vocab_mask"], b.want["vocab_mask"]) and np.array_equal(got["logits"], b.want["logits"])
                    else:
                        compare_step(dict(got, logits=b.want["logits"]) if kind == "host" else got, b.want, V)
                kept = [[None if t is None else t.clone() for t in results] for results in now]
                continue
            for results, first in zip(now, kept):
                for got, want in zip(results, first):
                    # (a row's slot in its group is dealt by atomics, and the order of its sums with it: full log-probabilities to 1e-4)
                    assert got is None or (torch.equal(got, want) if got.dtype == torch.int32 else bool(((got - want).abs() <= 1e-4).logical_or(got == want).all()))
