"""GPU: decode steps of fp32 dense models at few rows (the five-kernel chain and the cluster kernel) against the oracle, around
the sizes where its kernels change: row groups, weight rows longer than the registered pieces, key splits, passes of 256 keys."""
import pytest
import torch

from gpu_util import make_gpu_model, teacher_forced_compare
from paper_2608_12385_b200.inputs import make_tokens, make_weights, tiny_dense_fp32

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kw,B,T,npre", [
    (dict(), 1, 12, 9),                                             # rows below a group of four
    (dict(), 3, 20, 16),                                            # groups of eight, the last one partial
    (dict(), 16, 6, 4),                                             # 32 rows, the most of this chain
    (dict(), 17, 6, 4),                                             # one more: the generic chain
    (dict(), 2, 132, 125),                                          # from one split to two
    (dict(n_q_heads=2, n_kv_heads=1, head_dim=128, d_ff=1032), 1, 700, 697),  # several splits, long weight rows
    (dict(n_q_heads=4, n_kv_heads=1, final_norm=0), 2, 40, 36),     # four heads per KV head, no final norm
    (dict(n_paths=4, n_kv_heads=2), 3, 24, 20),                     # three branches
    (dict(n_paths=3, n_kv_heads=2), 2, 24, 20),                     # six rows of three paths through the cluster kernel
    (dict(d_ff=1024), 2, 24, 20),                                   # matrices beyond the cluster's shared memory
    (dict(d_model=128, n_q_heads=6, n_kv_heads=2, d_ff=192), 4, 24, 20),  # a slice over Q and K, eight rows
])
def test_few_row_decode_matches_the_oracle(kw, B, T, npre):
    cfg = tiny_dense_fp32().replace(n_layers=2, vocab=1003, **kw)
    w = make_weights(cfg, seed=31)
    teacher_forced_compare(cfg, w, make_tokens(cfg, B, T, seed=32), n_prefill=npre, grouped=True)


def test_few_row_attention_over_passes_of_256_keys_does_not_depend_on_the_splits():
    """At batch 16 a pair has few splits and each walks several passes; alone it has 16: same values to rounding."""
    cfg = tiny_dense_fp32().replace(n_layers=1, n_q_heads=16, n_kv_heads=16)
    w = make_weights(cfg, seed=33)
    tok = make_tokens(cfg, 16, 2, seed=34).cuda()
    a, b = make_gpu_model(cfg, w, 16, 2100), make_gpu_model(cfg, w, 1, 2100)
    gen = torch.Generator(device="cuda").manual_seed(3)
    k = torch.empty(1, 16, 2050, cfg.kv_dim, device="cuda").normal_(generator=gen)
    v = torch.empty_like(k).normal_(generator=gen)
    a.write_kv(k, v)
    b.write_kv(k[:, 5:6], v[:, 5:6])
    za, zb = a.decode_full(tok[:, 0].contiguous()), b.decode_full(tok[5:6, 0].contiguous())
    for name in ("z1", "z2"):  # sums of 2051 products in another order: a few 1e-6 relative
        torch.testing.assert_close(za[name][5:6], zb[name], rtol=1e-4, atol=2e-5)
