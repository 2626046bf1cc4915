"""The o projection's slices wait for every KV group they read, whatever the group's width: wider than
a 256-feature slice (several slices read one group), straddling slices, or narrower."""
import dataclasses

import numpy as np
import pytest

from paper_2607_12422_gb300 import pbd, synth


@pytest.mark.parametrize("hq,hkv,d", [(16, 8, 128), (16, 4, 128), (16, 2, 128), (12, 4, 128), (12, 4, 64), (24, 8, 64),
                                      (8, 8, 64), (20, 4, 64)])
@pytest.mark.parametrize("kind", [0, 1, 2])
def test_o_slices_wait_for_every_group_they_read(hq, hkv, d, kind):
    S = dataclasses.replace(synth.QWEN3_0_6B, n_layers=2, n_q_heads=hq, n_kv_heads=hkv, head_dim=d, vocab=4096)
    cfg = pbd.make_config(S, 16, 2, 600)
    items, _ = pbd.pbd_plan_pass(cfg, kind, [300, 40], 64, 152)
    op, lin, layer = items[:, 0] & 0xFF, (items[:, 0] >> 8) & 0xFF, items[:, 0] >> 16
    for l in range(2):
        att = items[(op == 2) & (layer == l)]
        for it in items[(op == 1) & (lin == 1) & (layer == l)]:
            heads = range(it[2] * 256 // d, ((it[2] + 1) * 256 - 1) // d + 1)
            groups = {h // (hq // hkv) for h in heads}
            counted = att[att[:, 6] == it[4]]
            assert groups <= set(counted[:, 2]), (l, it[2])
            assert it[5] == len(counted)  # every merge of both sequences (their items fit one wave)
