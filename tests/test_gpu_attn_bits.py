"""GPU: the bits that decode steps leave.  The order in which the attention adds -- a chain of products per 16 keys, the four warps'
states as (0 + 2) + (1 + 3), the partials of a pair eight at a time -- decides near-ties between tokens, so it stays as it is
whatever the code around it becomes.

Recorded on a B200, library built with nvcc 12.9.  Weights, cache and tokens are whole numbers times powers of two (torch's integer
draws), so that they are the same on every host; another compiler may contract other products and sums."""
import hashlib

import pytest
import torch

from gpu_util import make_gpu_model
from paper_2608_12385_b200.inputs import ModelConfig, make_tokens, make_weights

pytestmark = pytest.mark.gpu


def cfg_of(**kw):
    base = dict(d_model=256, n_layers=2, n_q_heads=8, n_kv_heads=8, head_dim=64, d_ff=512, vocab=512, weight_dtype="bf16")
    base.update(kw)
    return ModelConfig(**base)


def integers(like: torch.Tensor, gen: torch.Generator, unit: float, centre: float = 0.0) -> torch.Tensor:
    """Draws of -128..127 times a power of two: exact in bf16, about as wide as a normal draw of 74 units."""
    return (torch.randint(-128, 128, like.shape, generator=gen, dtype=torch.int32).float() * unit + centre).to(like.dtype)


def integer_weights(cfg: ModelConfig, seed: int) -> dict:
    gen = torch.Generator().manual_seed(seed)
    w = make_weights(cfg, seed=0)

    def draw(name, t):
        if name.endswith("_g"):  # norm gains around one
            return integers(t, gen, 2.0 ** -12, 1.0)
        if name.startswith("coup"):
            return integers(t, gen, 2.0 ** -7)
        return integers(t, gen, 2.0 ** -10)

    out = {n: draw(n, t) for n, t in w.items() if n != "layers"}
    out["layers"] = [{n: draw(n, t) for n, t in lw.items()} for lw in w["layers"]]
    return out


def digest(cfg: ModelConfig, lens: list, grouped: bool) -> str:
    """Of the logits, the next tokens and the whole cache of three steps."""
    gen = torch.Generator().manual_seed(62)
    B, T = len(lens), max(lens)
    cache = torch.empty(cfg.n_layers, B, T, cfg.kv_dim, dtype=cfg.torch_dtype)
    k, v = integers(cache, gen, 2.0 ** -6), integers(cache, gen, 2.0 ** -6)
    tok = make_tokens(cfg, B, 3, seed=63)
    gm = make_gpu_model(cfg, integer_weights(cfg, 61), B, T + 4)
    gm.write_kv(k, v)
    gm.set_seq_lens(lens)
    h = hashlib.sha256()
    for t in range(3):
        out = gm.decode_full(tok[:, t].cuda().contiguous(), grouped=grouped)
        for name in ("z1", "z2", "next") if grouped else ("z1", "next"):
            h.update(out[name].contiguous().cpu().numpy().tobytes())
    h.update(gm.kv_pool.view(torch.int16).cpu().numpy().tobytes())
    assert gm.sync_status() == (0, 0)
    return h.hexdigest()[:16]


CASES = [
    # more than eight stacked rows, ragged: several segments per CTA at d_h 64 and 128, three branches, sixteen query rows
    ("ragged64", cfg_of(), [1 + (37 * i) % 700 for i in range(100)]),
    ("ragged128", cfg_of(n_q_heads=16, head_dim=128), [60 + 11 * i for i in range(64)]),
    ("branches", cfg_of(n_q_heads=16, n_paths=4), [500 - 5 * i for i in range(60)]),
    ("sixteen", cfg_of(n_q_heads=32, n_kv_heads=4), [(i * i) % 900 + 5 for i in range(117)]),
    # one CTA per SM, a pair each
    ("deep64", cfg_of(), [100 + 50 * i for i in range(16)]),
    ("deep128", cfg_of(n_q_heads=16, head_dim=128), [1000 + 57 * i for i in range(16)]),
    # pairs split over many CTAs
    ("split", cfg_of(n_kv_heads=2, head_dim=128), [2400, 3000, 4090, 18500, 77]),
    # few rows on the chain that sums split-K partials: a mixture of experts, a width not in whole 64-element columns
    ("experts", cfg_of(n_kv_heads=2, head_dim=128, d_ff=0, n_experts=8, d_expert=128, k_primary=2, k_branch=2, n_shared_experts=1),
     [2400, 3000, 33]),
    ("narrow", cfg_of(d_ff=712), [700, 300]),
]
RECORDED = {  # grouped steps, primary-only steps
    "ragged64": ("3490384381808481", "bab24b3ad9235203"),
    "ragged128": ("2992fd839c73b7eb", "65d380c8fb6ba3c0"),
    "branches": ("3310bf5312481a35", "caa5cf6de46afaa0"),
    "sixteen": ("f3aebb257f250b74", "6622d4f952134afb"),
    "deep64": ("f0fe60fdf22d0cf6", "e996047af4f61d31"),
    "deep128": ("2de9935aed996475", "76ef4eb9c8a6c27c"),
    "split": ("12c2b8fd778b6533", "0326940b6eb8b642"),
    "experts": ("ad11f175014e018a", "d883ea5a47f40fa8"),
    "narrow": ("0690c3072c301f01", "c46571b73f40a5c9"),
}


@pytest.mark.parametrize("grouped", [True, False])
@pytest.mark.parametrize("name,cfg,lens", CASES, ids=[c[0] for c in CASES])
def test_decode_steps_leave_the_recorded_bits(name, cfg, lens, grouped):
    assert digest(cfg, lens, grouped) == RECORDED[name][0 if grouped else 1]
