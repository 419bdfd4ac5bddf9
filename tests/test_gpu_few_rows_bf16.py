"""GPU: decode steps of bf16 dense models at up to eight stacked rows (dbt_few.cuh) against the oracle, around the sizes where the
kernels change: room for 2, 4 or 8 rows, feature tiles of 16 (8 of gate and up) and stages of 512 elements that end early, rows
that stay in shared memory or pass through the ring, several tiles per CTA, and the splits of the attention behind them."""
import pytest
import torch

import oracle
from gpu_util import assert_logits_close, make_gpu_model, teacher_forced_compare
from paper_2608_12385_b200.inputs import ModelConfig, make_tokens, make_weights

pytestmark = pytest.mark.gpu


def cfg_of(**kw):
    base = dict(d_model=256, n_layers=3, n_q_heads=8, n_kv_heads=2, head_dim=64, d_ff=704, vocab=1003, weight_dtype="bf16")
    base.update(kw)
    return ModelConfig(**base)


@pytest.mark.parametrize("kw,B,T,npre", [
    (dict(), 1, 24, 20),                                                    # two rows
    (dict(n_paths=3), 1, 24, 20),                                           # three rows in room for four
    (dict(), 2, 24, 20),                                                    # four
    (dict(n_paths=5, n_q_heads=4), 1, 24, 20),                              # five in room for eight
    (dict(n_paths=3), 2, 24, 20),                                           # six, two branches
    (dict(), 4, 24, 20),                                                    # eight, the most
    (dict(), 5, 24, 20),                                                    # one sequence more: the other chain
    (dict(d_ff=712), 2, 24, 20),                                            # not in whole 64-element columns: the other chain
    (dict(d_model=1088, d_ff=576, n_layers=2), 1, 20, 17),                  # a third stage of one column
    (dict(d_model=128, n_q_heads=2, n_kv_heads=1, head_dim=128, d_ff=64, vocab=777), 3, 20, 17),  # less than one stage
    (dict(d_ff=6592, n_layers=2), 1, 12, 9),                                # 13 stages; two tiles of gate and up per CTA and more
    (dict(d_ff=6592, n_layers=2), 4, 12, 9),
    (dict(d_model=3584, d_ff=256, n_layers=2, vocab=5003), 1, 10, 8),       # rows of 28 KB stay, those of four rows do not
    (dict(d_model=3584, d_ff=256, n_layers=2, vocab=5003), 2, 10, 8),
    (dict(final_norm=0), 1, 20, 17),
    (dict(), 1, 132, 126),                                                  # from two stages of keys to three
    (dict(), 2, 1030, 1022),                                                # from sixteen to seventeen: the shortest segment grows
    (dict(n_paths=4), 2, 530, 526),
])
def test_few_row_decode_matches_the_oracle(kw, B, T, npre):
    cfg = cfg_of(**kw)
    w = make_weights(cfg, seed=31, matrix_std=0.05 if cfg.d_model <= 256 else 0.02)
    gm, _ = teacher_forced_compare(cfg, w, make_tokens(cfg, B, T, seed=32), n_prefill=npre, grouped=True)
    assert gm.sync_status() == (0, 0)


@pytest.mark.parametrize("paths,B", [(2, 1), (3, 1), (2, 4)])
def test_few_row_primary_only_steps_write_the_same_bits(paths, B):
    """Room and tiles follow the rows of all paths, so both modes add the same products in the same order."""
    cfg = cfg_of(n_paths=paths)
    w = make_weights(cfg, seed=33, matrix_std=0.05)
    tok = make_tokens(cfg, B, 300, seed=34).cuda()
    a, b = make_gpu_model(cfg, w, B, 300), make_gpu_model(cfg, w, B, 300)
    for m in (a, b):
        m.prefill(tok[:, :290].contiguous())
    for t in range(290, 300):
        x, y = a.decode_full(tok[:, t].contiguous()), b.decode_full(tok[:, t].contiguous(), grouped=False)
        assert torch.equal(x["z1"], y["z1"])
    for p, q in zip(a.export_kv(B, 300), b.export_kv(B, 300)):
        assert torch.equal(p.view(torch.int16), q.view(torch.int16))


# Two sixteens of weight rows per tile: from five rows and a contracted width of 4096 on, with enough tiles.  Here all four matrices of a
# layer and the output matrix take them: contracted widths of 4160, 4608 and 5184 end a stage early, gate and up have 324 tiles of 32
# rows and the output matrix 304, so that CTAs walk a second tile; the output matrix's last tile holds 11 rows (its second
# sixteen none) or 19.
LONG = dict(d_model=4160, n_q_heads=36, n_kv_heads=12, head_dim=128, d_ff=5184)


@pytest.mark.parametrize("paths,B,vocab", [(2, 4, 9707), (2, 3, 9715), (3, 2, 9707), (5, 1, 9715),
                                           (2, 2, 9707)])  # four rows: one sixteen per tile
def test_two_sixteens_of_weight_rows_per_tile_match_the_oracle(paths, B, vocab):
    cfg = cfg_of(n_paths=paths, n_layers=1, vocab=vocab, **LONG)
    gm, _ = teacher_forced_compare(cfg, make_weights(cfg, seed=37), make_tokens(cfg, B, 5, seed=38), n_prefill=2, grouped=True)
    assert gm.sync_status() == (0, 0)


def test_two_sixteens_per_tile_give_the_same_bits_grouped_and_primary_only():
    cfg = cfg_of(n_layers=2, vocab=9707, **LONG)
    w = make_weights(cfg, seed=39)
    tok = make_tokens(cfg, 4, 12, seed=40).cuda()
    a, b = make_gpu_model(cfg, w, 4, 12), make_gpu_model(cfg, w, 4, 12)
    for m in (a, b):
        m.prefill(tok[:, :9].contiguous())
    for t in range(9, 12):
        x, y = a.decode_full(tok[:, t].contiguous()), b.decode_full(tok[:, t].contiguous(), grouped=False)
        assert torch.equal(x["z1"], y["z1"])
    for p, q in zip(a.export_kv(4, 12), b.export_kv(4, 12)):
        assert torch.equal(p.view(torch.int16), q.view(torch.int16))


@pytest.mark.parametrize("knob,value", [("DBT_READOUT", "row"), ("DBT_EVICT_FIRST", "0"), ("DBT_GRAPH", "0"), ("DBT_PDL", "0")])
def test_few_row_steps_under_the_launch_knobs(monkeypatch, knob, value):
    """Without eviction hints, graph replay or programmatic launch (whose early page requests then wait too): the same step, also
    behind a prompt whose boundary rows rode along."""
    monkeypatch.setenv(knob, value)
    cfg = cfg_of()
    w = make_weights(cfg, seed=5, matrix_std=0.05)
    for grouped in (True, False):
        teacher_forced_compare(cfg, w, make_tokens(cfg, 3, 294, seed=6), n_prefill=290, grouped=grouped)
    tok = make_tokens(cfg, 2, 302, seed=7)
    om, gm = oracle.OracleModel(cfg, w, 2, 302), make_gpu_model(cfg, w, 2, 302)
    om.prefill(tok[:, :300].numpy(), want_logits=False)
    got = [gm.prefill_boundary(tok[:, :301].cuda().contiguous()), gm.decode_full(tok[:, 301].cuda().contiguous())]
    for t, g in zip((300, 301), got):
        want = om.decode_step(tok[:, t].numpy())
        for name in ("z1", "z2"):
            assert_logits_close(g[name], want[name], cfg.weight_dtype, f"position {t} {name}")
    assert gm.sync_status() == (0, 0)
