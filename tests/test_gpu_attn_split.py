"""GPU: how the decode attention deals its work when every CTA has several (sequence, KV head) pairs -- rows by falling
length, every second round backwards, an incomplete last round cut to fill the CTAs -- against the oracle on sampled rows."""
import numpy as np
import pytest
import torch

import oracle
from gpu_util import assert_logits_close, make_gpu_model
from paper_2608_12385_b200.inputs import ModelConfig, make_synthetic_kv, make_tokens, make_weights

pytestmark = pytest.mark.gpu


def cfg_of(**kw):
    base = dict(d_model=256, n_layers=2, n_q_heads=8, n_kv_heads=8, head_dim=64, d_ff=512, vocab=512, weight_dtype="bf16")
    base.update(kw)
    return ModelConfig(**base)


@pytest.mark.parametrize("cfg,lens", [
    (cfg_of(), [300] * 117),                                             # equal pairs, 3.2 per CTA
    (cfg_of(), [1 + (37 * i) % 700 for i in range(100)]),                # ragged, from one position on
    (cfg_of(head_dim=128, n_q_heads=16), [60 + 11 * i for i in range(64)]),
    (cfg_of(n_q_heads=16, n_kv_heads=8, n_paths=4), [500 - 5 * i for i in range(60)]),  # eight query rows, three branches
    (cfg_of(n_q_heads=16, n_kv_heads=2, n_layers=1), [(i * i) % 900 + 5 for i in range(128)]),  # the 16-row form, pairs < CTAs
])
def test_dealt_pairs_match_the_oracle_on_sampled_sequences(cfg, lens):
    B, T = len(lens), max(lens)
    w = make_weights(cfg, seed=41, matrix_std=0.05)
    k, v = make_synthetic_kv(cfg, B, T, seed=42)
    tok = make_tokens(cfg, B, 2, seed=43)
    gm = make_gpu_model(cfg, w, B, T + 4)
    gm.write_kv(k, v)
    gm.set_seq_lens(lens)
    pick = [0, 1, B // 2, B - 1]
    out = []
    for t in range(2):
        out.append(gm.decode_full(tok[:, t].cuda().contiguous()))
    for b in pick:
        om = oracle.OracleModel(cfg, w, 1, T + 4)
        om.inject_kv(k[:, b:b + 1, :lens[b]].float().numpy(), v[:, b:b + 1, :lens[b]].float().numpy(), lens[b])
        for t in range(2):
            o = om.decode_step(tok[b:b + 1, t].numpy())
            assert_logits_close(out[t]["z1"][b:b + 1], o["z1"], "bf16", f"row {b} step {t} z1")
            z2 = out[t]["z2"][b:b + 1] if cfg.n_paths == 2 else out[t]["z2"][:, b:b + 1]
            assert_logits_close(z2, np.asarray(o["z2"]).reshape(z2.shape), "bf16", f"row {b} step {t} z2")
    assert gm.sync_status() == (0, 0)


def test_dealt_pairs_grouped_and_primary_only_write_the_same_cache():
    cfg = cfg_of()
    lens = [200 + (53 * i) % 400 for i in range(110)]
    w = make_weights(cfg, seed=44, matrix_std=0.05)
    k, v = make_synthetic_kv(cfg, len(lens), max(lens), seed=45)
    tok = make_tokens(cfg, len(lens), 1, seed=46)[:, 0].cuda().contiguous()
    caches = []
    for grouped in (True, False):
        gm = make_gpu_model(cfg, w, len(lens), max(lens) + 4)
        gm.write_kv(k, v)
        gm.set_seq_lens(lens)
        gm.decode_full(tok, grouped=grouped)
        caches.append(gm.kv_pool.clone())
    assert torch.equal(caches[0], caches[1])


@pytest.mark.parametrize("heads,kv_heads,dh,paths", [(2, 2, 64, 2), (8, 2, 64, 2), (4, 2, 128, 2), (4, 2, 128, 3), (8, 2, 128, 2)])
def test_merge_of_many_segments_at_few_and_more_query_rows(heads, kv_heads, dh, paths):
    """2 to 8 query rows: one 16-byte piece of the output per thread (sixteen partials at once) up to 4 rows at d_h 128 or 8 at
    64, two pieces above; 40 segments (of 256 positions) go through groups, 10 through one merge."""
    cfg = cfg_of(n_q_heads=heads, n_kv_heads=kv_heads, head_dim=dh, n_paths=paths)
    test_dealt_pairs_match_the_oracle_on_sampled_sequences(cfg, [10250, 2570])


@pytest.mark.parametrize("kw,lens", [
    (dict(n_q_heads=8, n_kv_heads=2, head_dim=128), [2400, 3000, 4090]),       # 8 query rows against 4: nine to sixteen segments
    (dict(n_q_heads=8, n_kv_heads=2, head_dim=128), [18500]),                  # 72 segments: more than eight groups
    (dict(n_q_heads=4, n_kv_heads=2, head_dim=128, n_paths=3), [3600, 2500]),  # 6 against 2
    (dict(n_q_heads=16, n_kv_heads=2, head_dim=64), [19000, 2700]),            # 16 against 8 at d_h 64
])
def test_merge_of_many_segments_is_the_same_bits_grouped_and_primary_only(kw, lens):
    """The primary path must not depend on the step's mode.  How many partials a thread keeps in flight does, so the merge's
    rounding must not follow it.  Segments are of 256 positions here; three layers and four steps, so that a differing bit
    reaches the cache."""
    cfg = cfg_of(n_layers=3, **kw)
    w = make_weights(cfg, seed=47, matrix_std=0.05)
    k, v = make_synthetic_kv(cfg, len(lens), max(lens), seed=48)
    tok = make_tokens(cfg, len(lens), 4, seed=49)
    kv, z1 = [], []
    for grouped in (True, False):
        gm = make_gpu_model(cfg, w, len(lens), max(lens) + 8)
        gm.write_kv(k, v)
        gm.set_seq_lens(lens)
        z1.append([gm.decode_full(tok[:, t].cuda().contiguous(), grouped=grouped)["z1"] for t in range(4)])
        kv.append(gm.kv_pool.clone())
    assert torch.equal(kv[0], kv[1])
    assert all(torch.equal(a, b) for a, b in zip(*z1))


@pytest.mark.parametrize("kw", [dict(), dict(head_dim=128, n_q_heads=16), dict(n_q_heads=32, n_kv_heads=4)])  # (the last: 16 query rows)
def test_stages_that_segments_wrote_take_the_next_segments_pages(kw):
    """Several segments per CTA, whose last stages hold zeros, the new row and (up to eight query rows) the warps' states when the
    next segment's pages arrive in them: what the first sequences give is right, and twenty runs leave the same bits."""
    cfg = cfg_of(**kw)
    lens = [17 + (53 * i) % 650 for i in range(117)]
    test_dealt_pairs_match_the_oracle_on_sampled_sequences(cfg, lens)
    w = make_weights(cfg, seed=41, matrix_std=0.05)
    k, v = make_synthetic_kv(cfg, len(lens), max(lens), seed=42)
    tok = make_tokens(cfg, len(lens), 1, seed=43)[:, 0].cuda().contiguous()
    gm = make_gpu_model(cfg, w, len(lens), max(lens) + 4)
    gm.write_kv(k, v)
    first = None
    for _ in range(20):
        gm.set_seq_lens(lens)
        out = gm.decode_full(tok)
        got = [out["z1"].clone(), out["z2"].clone(), gm.kv_pool.clone()]
        first = first or got
        assert all(torch.equal(a, b) for a, b in zip(first, got))
