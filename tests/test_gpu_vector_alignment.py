"""GPU: norm gains, couplings and gates are plain fp32 vectors of the caller: any 4-byte alignment, as when they lie one after the
other in one buffer.  Same bits as with aligned vectors, on every chain that reads them four at a time."""
import pytest
import torch

from paper_2608_12385_b200 import binding
from paper_2608_12385_b200.inputs import ModelConfig, make_tokens, make_weights, tiny_dense_fp32
from test_gpu_parity import small_moe

pytestmark = pytest.mark.gpu


def off_by(t: torch.Tensor, n: int) -> torch.Tensor:
    """The same values n elements behind a 16-byte boundary."""
    buf = torch.empty(t.numel() + 4, dtype=t.dtype, device=t.device)
    return buf[n:n + t.numel()].copy_(t)


@pytest.mark.parametrize("cfg,B,n", [
    (tiny_dense_fp32().replace(n_layers=2), 2, 1),                 # the cluster kernel
    (tiny_dense_fp32().replace(n_layers=2, d_ff=1024), 2, 1),      # five kernels per layer, weight rows beyond the registered pieces
    (ModelConfig(d_model=256, n_layers=2, n_q_heads=8, n_kv_heads=2, head_dim=64, d_ff=712, vocab=1028, weight_dtype="bf16"), 70, 1),
    (ModelConfig(d_model=256, n_layers=2, n_q_heads=8, n_kv_heads=2, head_dim=64, d_ff=712, vocab=500, weight_dtype="bf16"), 1, 300),
    (small_moe(), 1, 300),
    (small_moe(n_shared_experts=0, compute_matched=1), 1, 300),
])
def test_unaligned_vectors_give_the_same_bits(cfg, B, n):
    wd = binding.weights_to_device(make_weights(cfg, seed=51, matrix_std=0.05))
    moved = {**wd, "layers": [{k: off_by(v, 1 + i % 3) if v.dim() == 1 else v for i, (k, v) in enumerate(lw.items())} for lw in wd["layers"]]}
    for k in ("embed_norm_g", "final_norm_g"):
        moved[k] = off_by(wd[k], 3)
    assert any(v.data_ptr() % 16 for v in moved["layers"][0].values())
    tok = make_tokens(cfg, B, n + 2, seed=52).cuda()
    out = []
    for w in (wd, moved):
        gm = binding.Model(cfg, w, B, n + 2)
        z = [gm.prefill(tok[:, :n].contiguous(), want_logits=True)]
        for t in range(2):
            g = gm.decode_full(tok[:, n + t].contiguous())
            z += [g["z1"].clone(), g["z2"].clone()]
        assert gm.sync_status() == (0, 0)
        out.append((z, gm.kv_pool.clone()))
    assert all(torch.equal(a, b) for a, b in zip(out[0][0], out[1][0])) and torch.equal(out[0][1], out[1][1])
