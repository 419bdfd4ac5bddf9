"""GPU: prompt chunks at the edges of the paired-SM GEMMs' 256 x 256 tiles and of the prompt attention's 128-row query
and 128-key tiles, against the oracle's position-by-position primary pass."""
import numpy as np
import pytest
import torch

import oracle
from gpu_util import assert_logits_close, make_gpu_model
from paper_2608_12385_b200.inputs import ModelConfig, make_tokens, make_weights

pytestmark = pytest.mark.gpu


def cfg_of(**kw):
    base = dict(d_model=256, n_layers=2, n_q_heads=8, n_kv_heads=2, head_dim=64, d_ff=712, vocab=500, weight_dtype="bf16")
    base.update(kw)
    return ModelConfig(**base)


@pytest.mark.parametrize("cfg,B,n,past", [
    (cfg_of(), 1, 257, 0),                                       # one row past a row tile
    (cfg_of(), 1, 512, 0),                                       # whole row tiles, whole key tiles
    (cfg_of(), 2, 300, 0),                                       # a row tile that spans two sequences
    (cfg_of(), 1, 300, 133),                                     # behind a cached prefix that ends inside a page
    (cfg_of(d_model=328, d_ff=1032), 1, 385, 0),                 # ragged feature tiles in every matrix
    (cfg_of(n_q_heads=2, n_kv_heads=2), 1, 400, 0),              # one head per KV head: 128 positions per query tile
    (cfg_of(n_q_heads=16, n_kv_heads=2, n_layers=1), 3, 130, 1),  # eight heads per KV head: 16 positions per query tile
    (cfg_of(n_q_heads=4, n_kv_heads=2, head_dim=128, n_layers=1), 1, 650, 0),
    (cfg_of(n_layers=1), 32, 640, 0),                            # a chunk of 18944 rows and one of 1504
])
def test_prompt_chunk_edges_match_the_oracle(cfg, B, n, past, std=0.05):
    w = make_weights(cfg, seed=91, matrix_std=std)
    total = past + n
    tok = make_tokens(cfg, B, total, seed=92)
    om = oracle.OracleModel(cfg, w, B, total)
    gm = make_gpu_model(cfg, w, B, total)
    want = om.prefill(tok.numpy())
    if past:
        gm.prefill(tok[:, :past].cuda().contiguous())
    # logits are the last position's own pass; n - 1 positions go through as one chunk
    got = gm.prefill(tok[:, past:].cuda().contiguous(), want_logits=True)
    assert_logits_close(got, want, "bf16", "prompt logits")
    k_dev, v_dev = gm.export_kv(B, total)
    # bf16 storage (2^-9 relative) on top of the logit-level error of fp32 sums
    np.testing.assert_allclose(k_dev.float().numpy(), om.k_cache[:, :B, :total], rtol=2.0 ** -8, atol=5e-3)
    np.testing.assert_allclose(v_dev.float().numpy(), om.v_cache[:, :B, :total], rtol=2.0 ** -8, atol=5e-3)
    assert gm.sync_status() == (0, 0)


@pytest.mark.parametrize("cfg,B,n,past", [
    (cfg_of(), 1, 129, 0),                                        # 128 rows: the most of the short form
    (cfg_of(), 1, 130, 0),                                        # one row more
    (cfg_of(), 1, 100, 1),                                        # behind one cached position: the other kernel
    (cfg_of(), 1, 3, 0),                                          # two positions
    (cfg_of(), 4, 33, 0),                                         # 4 x 32 rows, whole pages
    (cfg_of(), 3, 18, 0),
    (cfg_of(n_q_heads=2, n_kv_heads=2, head_dim=128), 1, 100, 0),  # one head per KV head: 128 positions per block
    (cfg_of(n_q_heads=8, n_kv_heads=1, head_dim=128), 2, 50, 0),   # eight: 16 positions per block
    (cfg_of(n_q_heads=16, n_kv_heads=2, n_layers=1), 1, 90, 0),
])
def test_short_prompts_match_the_oracle(cfg, B, n, past):
    """First chunks of at most 128 rows, around the edges of their eight 16-row query tiles and 64-key stages."""
    test_prompt_chunk_edges_match_the_oracle(cfg, B, n, past)


def test_a_captured_short_prompt_replayed_behind_a_longer_cache():
    """The short form is chosen from the lengths that the host knows when the call is made; a replay of the captured call works on
    the device's lengths, whatever they are by then."""
    from paper_2608_12385_b200 import binding
    from paper_2608_12385_b200.inputs import make_synthetic_kv
    cfg = cfg_of()
    w = make_weights(cfg, seed=99, matrix_std=0.05)
    tok = make_tokens(cfg, 1, 40, seed=100)
    k, v = make_synthetic_kv(cfg, 1, 300, seed=101)
    dev = tok.cuda().contiguous()
    stream = torch.cuda.Stream()
    gm = binding.Model(cfg, binding.weights_to_device(w), 1, 400, stream=stream)
    gm.prefill(dev)
    torch.cuda.synchronize()
    gm.reset()
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream):
        gm.prefill(dev)
    gm.import_kv(k, v)  # the capture ran nothing: 300 positions, as the replay finds them
    graph.replay()
    torch.cuda.synchronize()
    om = oracle.OracleModel(cfg, w, 1, 400)
    om.inject_kv(k.float().numpy(), v.float().numpy(), 300)
    om.prefill(tok.numpy())
    gm.set_seq_lens([340])
    k_dev, v_dev = gm.export_kv(1, 340)
    np.testing.assert_allclose(k_dev.float().numpy(), om.k_cache[:, :1, :340], rtol=2.0 ** -8, atol=5e-3)
    np.testing.assert_allclose(v_dev.float().numpy(), om.v_cache[:, :1, :340], rtol=2.0 ** -8, atol=5e-3)
    assert gm.sync_status() == (0, 0)


def test_stale_pool_contents_behind_the_prompt_do_not_reach_it():
    """Pages past the last key hold whatever the pool held before; NaN there must change nothing."""
    cfg = cfg_of()
    w = make_weights(cfg, seed=93, matrix_std=0.05)
    for n in (333, 71):
        tok = make_tokens(cfg, 1, n, seed=94).cuda().contiguous()
        a, b = make_gpu_model(cfg, w, 1, 512), make_gpu_model(cfg, w, 1, 512)
        b.kv_pool.fill_(float("nan"))
        za, zb = a.prefill(tok, want_logits=True), b.prefill(tok, want_logits=True)
        assert torch.equal(za, zb) and torch.isfinite(za).all()
        assert torch.equal(a.export_kv(1, n)[0], b.export_kv(1, n)[0])


@pytest.mark.parametrize("kw,B,n,std", [
    (dict(n_experts=4, d_expert=200), 1, 700, 0.05),                                  # lists of several row tiles of an expert
    (dict(n_experts=64, d_expert=136, k_branch=2), 2, 150, 0.05),                     # short lists, some experts without a row
    (dict(n_experts=8, d_expert=328, n_shared_experts=0, k_branch=8), 1, 513, 0.05),  # no shared expert: the combine kernel
    (dict(n_experts=8, d_expert=128, n_shared_experts=2, k_primary=3, d_model=328), 1, 300, 0.05),
    (dict(n_experts=5, d_expert=264, k_primary=2), 1, 290, 0.05),                     # row tiles of 96 to 160 rows: a ring of five or six stages
    (dict(n_experts=67, d_expert=64, k_primary=3), 1, 260, 0.05),                     # a router row of 67 logits
    (dict(n_experts=8, d_expert=128), 32, 640, 0.05),                                 # a chunk of 18944 rows and one of 1536
    # rows of more than 8192 columns.  Logits are sums of d products of unit-scale states and weights of deviation std: the stated
    # tolerance is for std sqrt(d) = 0.05 sqrt(256) = 0.8, which at d = 8456 is std = 0.0087.
    (dict(n_experts=6, d_expert=64, d_model=8456, n_layers=1, n_q_heads=2), 1, 257, 0.0087),
])
def test_moe_prompt_chunk_edges_match_the_oracle(kw, B, n, std):
    from test_gpu_parity import small_moe, test_moe_prompt_chunks_of_more_than_one_row_tile_match_the_oracle as check
    check(small_moe(**kw), B, n, std)


def test_moe_prompt_chunks_take_the_same_kernels_at_any_number_of_experts():
    """A prompt of more than 256 rows goes through the paired-SM chain whether or not the experts come in fours."""
    from test_gpu_parity import small_moe
    names = {}
    for E in (5, 8):
        cfg = small_moe(n_experts=E)
        gm = make_gpu_model(cfg, make_weights(cfg, seed=97, matrix_std=0.05), 1, 400)
        gm.profile_begin()
        gm.prefill(make_tokens(cfg, 1, 300, seed=98).cuda().contiguous())
        names[E] = {(e["name"], e["launches"]) for e in gm.profile_end()}
    assert names[5] == names[8]
    assert ("expert_gateup", cfg.n_layers) in names[5] and not any(n.startswith("resid") for n, _ in names[5])


@pytest.mark.parametrize("n_out,K,R", [(2048, 2048, 256), (1028, 520, 129), (4096, 2816, 234), (1024, 64, 200), (11264, 2048, 130)])
def test_many_row_decode_widths_match_the_oracle(n_out, K, R):
    """Decode steps of 129 to 256 stacked rows take the paired-SM GEMMs (fewer: row tiles of 128 on one SM): tiles of 96 to 192
    features, unsplit and over three and four pairs of a cluster, ragged last k-tiles and feature tiles.  One layer whose MLP has
    the given widths (K = 2816: the down projection's, behind a d of 256), primary rows and branch rows."""
    cfg = cfg_of(d_model=K if K <= 2048 else 256, d_ff=max(n_out, 2 * K if K > 2048 else K) // 2 // 8 * 8, n_layers=1, vocab=1028)
    B = (R + 1) // 2
    w = make_weights(cfg, seed=95, matrix_std=0.02)
    tok = make_tokens(cfg, B, 3, seed=96)
    from gpu_util import teacher_forced_compare
    # tokens: logits may be off by the stated 2e-2 each, so two probabilities closer than e^(2 x 2e-2) - 1 may swap
    teacher_forced_compare(cfg, w, tok, n_prefill=1, grouped=True, token_margin=4.1e-2)


@pytest.mark.parametrize("model,B", [("1b", 66), ("1b", 117), ("8b", 70), ("moe", 75)])
def test_many_row_decode_at_the_presets_widths_on_sampled_sequences(model, B):
    """One layer of the presets at 132 to 234 stacked rows: tiles of 128 features over two pairs (1B and MoE Q|K|V, shared gate|up),
    of 192 over three (8B O and down), of 96 over three, and the unsplit output matrix in tiles of 256."""
    from paper_2608_12385_b200.inputs import PRESETS, make_synthetic_kv
    cfg = PRESETS[model]().replace(n_layers=1, **({"vocab": 8192} if model == "8b" else {}))
    w = make_weights(cfg, seed=0)
    lens = [3 + (11 * b) % 60 for b in range(B)]
    k, v = make_synthetic_kv(cfg, B, max(lens), seed=3)
    tok = make_tokens(cfg, B, 2, seed=2)
    gm = make_gpu_model(cfg, w, B, max(lens) + 4)
    gm.write_kv(k, v)
    gm.set_seq_lens(lens)
    out = []
    for t in range(2):
        out.append(gm.decode_full(tok[:, t].cuda().contiguous()))
        out[-1]["experts"] = gm.last_experts(B).numpy() if cfg.is_moe else None
    for b in (0, B // 2, B - 1):
        om = oracle.OracleModel(cfg, w, 1, max(lens) + 4)
        om.inject_kv(k[:, b:b + 1, :lens[b]].float().numpy(), v[:, b:b + 1, :lens[b]].float().numpy(), lens[b])
        for t in range(2):
            forced = np.ascontiguousarray(out[t]["experts"][:, :, b:b + 1]) if cfg.is_moe else None
            o = om.decode_step(tok[b:b + 1, t].numpy(), forced_experts=forced)
            assert_logits_close(out[t]["z1"][b:b + 1], o["z1"], "bf16", f"row {b} step {t} z1")
            assert_logits_close(out[t]["z2"][b:b + 1], o["z2"], "bf16", f"row {b} step {t} z2")
    assert gm.sync_status() == (0, 0)


@pytest.mark.parametrize("n", [201, 801])
def test_1b_width_prompts_of_a_few_row_tiles(n):
    """One layer of the 1B model at 200 and 800 rows: the residual GEMMs over three and four pairs per tile (192 and 256 features)
    and over two; Q|K|V split and unsplit."""
    from paper_2608_12385_b200.inputs import PRESETS
    test_prompt_chunk_edges_match_the_oracle(PRESETS["1b"]().replace(n_layers=1), 1, n, 0, std=0.02)


@pytest.mark.parametrize("kw,n", [
    (dict(n_q_heads=4, n_kv_heads=1, head_dim=64), 300),    # K and V share one tile of features
    (dict(n_q_heads=6, n_kv_heads=3, head_dim=64), 258),    # 192 features of each, one row in the second row tile
    (dict(n_q_heads=6, n_kv_heads=3, head_dim=128), 515),   # a tile and a half of each
    (dict(n_q_heads=4, n_kv_heads=2, head_dim=128), 90),    # a chunk on the decode step's GEMMs
])
def test_prompts_whose_outputs_nobody_reads_fill_the_whole_cache(kw, n):
    """The last layer of such a prompt forms keys and values alone; a decode step behind it sees them."""
    cfg = cfg_of(**kw)
    w = make_weights(cfg, seed=41, matrix_std=0.05)
    tok = make_tokens(cfg, 2, n + 1, seed=42)
    om = oracle.OracleModel(cfg, w, 2, n + 1)
    gm = make_gpu_model(cfg, w, 2, n + 1)
    om.prefill(tok[:, :n].numpy())
    gm.prefill(tok[:, :n].cuda().contiguous())
    want, got = om.decode_step(tok[:, n].numpy()), gm.decode_full(tok[:, n].cuda().contiguous())
    for name in ("z1", "z2"):
        assert_logits_close(got[name], want[name], cfg.weight_dtype, name)


@pytest.mark.parametrize("kw,B,S,past", [
    (dict(), 1, 160, 0),                                        # one sequence's rows behind 159
    (dict(), 1, 225, 0),                                        # the last group of the row tile (224 + 32 rows)
    (dict(), 1, 226, 0),                                        # no room in the row tile: the step runs by itself
    (dict(n_paths=3), 12, 30, 0),                               # 360 - 12 rows, two groups of ten sequences' three paths
    (dict(n_paths=4, n_q_heads=4, n_kv_heads=2), 9, 40, 0),     # eight sequences to a group
    (dict(n_layers=3), 20, 41, 0),                              # two paths of twenty sequences: the last layer on the wider chain
    (dict(n_layers=3), 2, 400, 133),                            # behind a cached prefix
    (dict(n_q_heads=4, n_kv_heads=2, head_dim=128, d_ff=704), 3, 300, 0),
    (dict(n_q_heads=16, n_kv_heads=2), 1, 333, 0),              # sixteen query rows per KV head
    (dict(d_model=328, d_ff=1032), 2, 150, 0),                  # ragged feature tiles
    (dict(n_q_heads=2, n_kv_heads=2, d_ff=2048, n_layers=2), 1, 650, 0),
])
def test_boundary_step_whose_rows_ride_in_the_prompts_last_chunk(kw, B, S, past):
    """The boundary evaluation, the cache it leaves and a step behind it against the oracle."""
    cfg = cfg_of(**kw)
    w = make_weights(cfg, seed=51, matrix_std=0.05)
    tok = make_tokens(cfg, B, past + S + 1, seed=52)
    om = oracle.OracleModel(cfg, w, B, past + S + 1)
    gm = make_gpu_model(cfg, w, B, past + S + 1)
    if past:
        gm.prefill(tok[:, :past].cuda().contiguous())
    om.prefill(tok[:, :past + S - 1].numpy(), want_logits=False)
    want = om.decode_step(tok[:, past + S - 1].numpy())
    got = gm.prefill_boundary(tok[:, past:past + S].cuda().contiguous())
    for name in ("z1", "z2"):
        assert_logits_close(got[name], want[name], cfg.weight_dtype, name)
    k_dev, v_dev = gm.export_kv(B, past + S)
    # the prompt's rows: one attention, whose queries and weights are bf16, lies before the second layer's keys and values, up to
    # 5e-3 as in the tests above; every further layer adds another one's.  The rows that rode: up to 5e-3 at any depth
    for got_kv, want_kv in ((k_dev.float().numpy(), om.k_cache[:, :B]), (v_dev.float().numpy(), om.v_cache[:, :B])):
        np.testing.assert_allclose(got_kv[:, :, past + S - 1], want_kv[:, :, past + S - 1], rtol=2.0 ** -8, atol=5e-3)
        for layer in range(cfg.n_layers):
            np.testing.assert_allclose(got_kv[layer], want_kv[layer, :, :past + S], rtol=2.0 ** -8, atol=5e-3 * max(layer, 1))
    want, got = om.decode_step(tok[:, past + S].numpy()), gm.decode_full(tok[:, past + S].cuda().contiguous())
    for name in ("z1", "z2"):
        assert_logits_close(got[name], want[name], cfg.weight_dtype, name)
    assert gm.sync_status() == (0, 0)
