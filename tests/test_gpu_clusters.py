"""Decode attention through thread-block clusters (small steps, no second
pass): every cluster shape the host picks (test_rules_cpu.py checks that these
steps pick it), rows that end on and around page
boundaries, rows with fewer pages than the cluster has warps, and rows that
outgrow what the shape was picked for, against the float64 oracle."""
import numpy as np
import pytest
import torch

import oracle
from paper_2603_12707_gb300 import kvdecode as kd
from paper_2603_12707_gb300 import workloads as wl
from paper_2603_12707_gb300.harness import DecodeSession

from _gpu_common import Tracked, assert_close, bf16_to_f64, u16

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("fused", [False, True])
@pytest.mark.parametrize("Hq,Hkv,d,lens", [
    (28, 4, 128, [2200, 33]),                       # 8 CTAs of 8 warps
    (14, 2, 64, [2300, 0]),
    (8, 8, 128, [700, 1, 16, 15]),                  # 8 of 4
    (56, 8, 128, [300, 511, 512]),
    (16, 16, 128, [300, 17, 0, 31, 250]),           # 4 of 4
    (24, 24, 64, [100, 64, 63, 1, 47]),            # 2 of 4
    (16, 8, 128, [90, 0, 15, 16, 47, 90, 3, 2, 77, 61, 33, 32]),
    (8, 8, 64, [60 - 3 * (b % 20) for b in range(24)]),   # 1 of 4
    (6, 2, 64, [40 - (b % 40) for b in range(120)]),
])
def test_cluster_shapes_match_the_oracle(kvlib, Hq, Hkv, d, lens, fused):
    cfg = wl.custom("cluster", 2, Hq, Hkv, d, len(lens), lens=lens, seed=91 + Hq + d, page_order="shuffled")
    t = Tracked(cfg, extra_tokens=8)
    n0 = t.sess.query().kernel_launches
    for _ in range(3):
        t.begin_step()
        for layer in range(cfg.num_layers):
            out, q, _, _ = t.run_layer(layer, fused=fused)
            torch.cuda.synchronize()
            ref, vmax = t.oracle(layer, q)
            assert_close(bf16_to_f64(out), ref, vmax, gqa=Hq > Hkv)
    # one step kernel and one attention launch per layer (and its append): no merge pass
    assert t.sess.query().kernel_launches - n0 == 3 * (1 + cfg.num_layers * (1 if fused else 2))
    t.close()


@pytest.mark.parametrize("Hq,Hkv,d", [(4, 4, 128), (14, 2, 64), (14, 2, 128)])   # a plan, and clusters of 64 warps
def test_rows_that_outgrow_the_shape_and_a_failed_row(kvlib, Hq, Hkv, d):
    """Device steps pick their clusters from the rows held when they are
    enabled (a page each); then a row grows to 9000 tokens, far past the
    page-id window of every warp.  A sequence id outside the cache gets no
    output."""
    lens = [5, 16, 3, 30]
    cfg = wl.custom("outgrow", 1, Hq, Hkv, d, 4, lens=lens, seed=17 + d)
    sess = DecodeSession(cfg, extra_tokens=9100)
    sess.fill_prefix()
    h = sess.h
    kd.kv_cache_device_steps(h, 4)
    gen = torch.Generator(device="cuda").manual_seed(3)
    rows = [[wl.kv_block(cfg, 0, b, n, kind, "cuda") for kind in "kv"] for b, n in enumerate(lens)]
    long = [torch.randn((9000, Hkv, d), generator=gen, device="cuda").bfloat16() for _ in "kv"]
    kd.kv_seq_reserve(h, sess.seq_ids[1], 9000)
    kd.kv_write_tokens(h, 0, sess.seq_ids[1], lens[1], 9000, long[0], long[1])
    rows[1] = [torch.cat(x) for x in zip(rows[1], long)]
    bad = list(sess.seq_ids)
    bad[2] = 99
    ids = torch.tensor(bad, dtype=torch.int32, device="cuda")
    q, kn, vn = wl.step_inputs(cfg, 0, 0, "cuda")
    out = torch.full_like(q, 7.0)
    kd.kv_begin_step_device(h, 4, ids)
    kd.decode_attention_append(h, 0, 4, q, kn, vn, out)
    torch.cuda.synchronize()
    assert kd.kv_cache_query(h, raise_on_device_error=False).device_error == kd.KVC_DEVERR_SEQ_RANGE
    assert bool((out[2] == 7.0).all())
    live = [0, 1, 3]
    k = [np.concatenate([u16(rows[b][0]), u16(kn[b:b + 1])]) for b in live]
    v = [np.concatenate([u16(rows[b][1]), u16(vn[b:b + 1])]) for b in live]
    ref = oracle.decode_attention(u16(q)[live], [len(x) for x in k], np.concatenate(k), np.concatenate(v))
    vmax = np.array([np.abs(oracle.bf16_to_f64(x)).max() for x in v])
    assert_close(bf16_to_f64(out)[live], ref, vmax, gqa=Hq > Hkv)
    sess.close()
