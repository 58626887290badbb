"""The dense expansion against the CPU oracle at the edges of its units (64 octets a warp), row groups (32 rows), class words (four at a
time where the masks' alignment allows) and plans; words past the row's last one stay untouched."""
import numpy as np
import pytest
import torch

import oracle
import synth
from synth import rng
from paper_2605_29986_b200 import binding as cz
from _gpu_util import Ctx, dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("V,K,B", [(1, 1, 1), (511, 128, 31), (512, 129, 32), (513, 127, 33), (8192, 1024, 65), (8224, 640, 7), (50001, 4097, 40),
                                   (130000, 20000, 3), (60000, 40000, 5), (32064, 300, 1030)])
@pytest.mark.parametrize("pad", [0, 1, 4])  # words between the rows of the masks: rows on 16-byte boundaries or not
def test_expand(V, K, B, pad):
    part = synth.zipf_partition(V, K, seed=V + K)
    KW, VW = (K + 31) // 32, (V + 31) // 32
    cm = np.full((B, KW + pad), 0xFFFFFFFF, dtype=np.uint32)
    cm[:, :KW] = synth.class_mask_bernoulli(K, B, 0.4, rng.stream_key(rng.SEED_BASE, 940, V, K))
    if K % 32:
        cm[:, KW - 1] |= np.uint32(0xFFFFFFFF) << np.uint32(K % 32)  # bits from K on are ignored
    d_vm = torch.full((B, VW + 1), 0x5A5A5A5A, dtype=torch.int32, device="cuda")
    with Ctx([part]) as ctx:
        cz.cfgzip_expand_mask(ctx.h, ctx.ids[0], None, dev(cm), cm.shape[1], d_vm, VW + 1, B, cz.DENSE)
        torch.cuda.synchronize()
    got = d_vm.cpu().numpy().view(np.uint32)
    assert np.array_equal(got[:, :VW], oracle.expand_mask(part.c, K, np.ascontiguousarray(cm[:, :KW])))
    assert (got[:, VW] == 0x5A5A5A5A).all()


@pytest.mark.parametrize("B", [3, 70])
def test_expand_and_map_rows_of_several_partitions(B):
    V = 9000
    parts = [synth.zipf_partition(V, k, seed=i) for i, k in enumerate((128, 333, 1000))]
    row_part = (np.arange(B) * 5 % 3).astype(np.int32)
    KW, VW = 32, (V + 31) // 32
    cm = synth.class_mask_bernoulli(1000, B, 0.3, rng.stream_key(rng.SEED_BASE, 941))
    want = np.stack([oracle.expand_mask(parts[p].c, parts[p].K, cm[b:b + 1])[0] for b, p in enumerate(row_part)])
    tok = (np.arange(B) * 37 % V).astype(np.int32)
    with Ctx(parts) as ctx:
        for rows in ("given", "planned"):
            d_rp = dev(row_part)
            if rows == "planned":
                cz.cfgzip_plan_rows(ctx.h, ctx.ids[0], d_rp, B)
                d_rp = cz.ROWS_AS_PLANNED
            d_vm = torch.zeros((B, VW), dtype=torch.int32, device="cuda")
            cz.cfgzip_expand_mask(ctx.h, ctx.ids[0], d_rp, dev(cm), KW, d_vm, VW, B, cz.DENSE)
            assert np.array_equal(d_vm.cpu().numpy().view(np.uint32), want), rows
        d_rep = torch.zeros(B, dtype=torch.int32, device="cuda")
        cz.cfgzip_map_tokens(ctx.h, ctx.ids[0], dev(row_part), dev(tok), d_rep, B)
        assert np.array_equal(d_rep.cpu().numpy(), np.array([parts[p].r[parts[p].c[t]] for p, t in zip(row_part, tok)]))
