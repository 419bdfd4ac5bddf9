"""Timing cases: what a program that serves a Decode-Branch model has this library do.

Two kinds of work, both through `paper_2608_12385_b200.binding.Model`:

- "decode": sequences with a cached context each take a few decode steps (grouped, or primary-only as the
  comparison path), the step's tokens supplied by the caller, as when a given continuation is scored; the logits of
  every step, the next tokens and alpha are kept.
- "prompt": `prefill_boundary` over whole prompts (from an empty cache, or behind a cached prefix), which fills the
  cache and makes the first mixture prediction.

Models are the package's own presets.  Weights, tokens and cached contexts are random draws of the distributions the
package's inputs module uses, made on the GPU.  Cached contexts lie in pages scattered over the pool.
"""
from __future__ import annotations

import torch

from paper_2608_12385_b200 import binding
from paper_2608_12385_b200.inputs import PRESETS, ModelConfig

PAGE = 16


def listed() -> list[dict]:
    return [
        # the smallest calls: a tiny fp32 model, two sequences; latency and launches are all there is
        {"name": "decode-tiny-fp32", "kind": "decode", "model": "tiny", "batch": 2, "ctx": 64, "steps": 16},
        # one interactive user of the 1B model: every weight streamed for two stacked rows
        {"name": "decode-1b-one-user", "kind": "decode", "model": "1b", "batch": 1, "ctx": 2048, "steps": 8},
        # the benchmark's own workload: a batch of 16 behind prompts of 2048
        {"name": "decode-1b-batch16", "kind": "decode", "model": "1b", "batch": 16, "ctx": 2048, "steps": 8},
        # a busy server: many sequences, every one at its own length
        {"name": "decode-1b-busy-ragged", "kind": "decode", "model": "1b", "batch": 117, "ctx": 1900, "ragged": True,
         "steps": 4},
        # long documents on the 8B-shaped model: the cache outweighs the matrices
        {"name": "decode-8b-long", "kind": "decode", "model": "8b", "batch": 4, "ctx": 32768, "steps": 4},
        # mixture of experts at a small batch, both paths with the same fan-out
        {"name": "decode-moe-batch8", "kind": "decode", "model": "moe", "batch": 8, "ctx": 4096, "steps": 4},
        # mixture of experts at a large batch with the widest branch fan-out: nearly every expert is loaded
        {"name": "decode-moe-batch32-wide", "kind": "decode", "model": "moe", "batch": 32, "ctx": 4096, "k_branch": 8,
         "steps": 4},
        # a short chat turn: the time to the first token
        {"name": "prompt-1b-short", "kind": "prompt", "model": "1b", "batch": 1, "ctx": 333},
        # a batch of full prompts, as the benchmark prefills them
        {"name": "prompt-1b-batch", "kind": "prompt", "model": "1b", "batch": 16, "ctx": 2048},
        # one long document into the 8B-shaped model
        {"name": "prompt-8b-long", "kind": "prompt", "model": "8b", "batch": 1, "ctx": 8192},
        # a batch of prompts into the mixture of experts
        {"name": "prompt-moe-batch", "kind": "prompt", "model": "moe", "batch": 32, "ctx": 1024},
    ]


def _log_int(rng, lo: int, hi: int) -> int:
    return min(hi, max(lo, int(round(lo * (hi / lo) ** rng.random()))))


def draw(rng) -> dict:
    kind = rng.choice(["decode", "decode", "prompt"])
    model = rng.choice(["tiny", "1b", "1b", "1b", "8b", "moe", "moe"])
    case = {"kind": kind, "model": model}
    if kind == "decode":
        batch_max, ctx_max, slots = {"tiny": (8, 2048, 8192), "1b": (128, 65536, 262144), "8b": (16, 32768, 131072),
                                     "moe": (32, 16384, 131072)}[model]
        case["batch"] = _log_int(rng, 1, batch_max)
        case["ctx"] = _log_int(rng, 16, min(ctx_max, slots // case["batch"]))
        case["steps"] = rng.randint(2, 4) if model != "tiny" else rng.randint(4, 16)
        case["ragged"] = rng.random() < 0.5
        case["primary_only"] = rng.random() < 0.25
    else:
        batch_max, ctx_max, slots = {"tiny": (8, 512, 1024), "1b": (32, 16384, 32768), "8b": (8, 8192, 8192),
                                     "moe": (32, 8192, 32768)}[model]
        case["batch"] = _log_int(rng, 1, batch_max)
        case["ctx"] = _log_int(rng, 32, min(ctx_max, slots // case["batch"]))
        # a further turn of a conversation: the prompt continues behind what the cache holds
        case["cached"] = rng.choice([0, 0, rng.randint(1, max(2, min(2 * case["ctx"], 4096)))])
    if model == "moe":
        case["k_branch"] = rng.choice([2, 4, 8])
        case["router_mode"] = rng.choice([0, 0, 1])
        case["compute_matched"] = rng.choice([0, 0, 1])
    else:
        case["paths"] = rng.choice([2, 2, 2, 3, 4])
        case["batch"] = min(case["batch"], 256 // case["paths"])  # a step holds at most 256 stacked rows
    return case


def _config(case: dict) -> ModelConfig:
    cfg = PRESETS[case["model"]]()
    keys = {"k_branch": "k_branch", "router_mode": "router_mode", "compute_matched": "compute_matched", "paths": "n_paths"}
    return cfg.replace(**{field: case[key] for key, field in keys.items() if key in case})


def _cached_lengths(case: dict) -> list[int]:
    """Positions that each sequence holds before the pass."""
    B = case["batch"]
    if case["kind"] == "prompt":
        return [case.get("cached", 0)] * B
    if not case.get("ragged"):
        return [case["ctx"] - 1] * B
    # spread from a sixteenth of the context to all of it, in no particular order
    lo, hi = max(1, case["ctx"] // 16), case["ctx"]
    return [lo + (hi - lo) * ((i * 37 + 11) % B) // max(1, B - 1) for i in range(B)]


def _weights(cfg: ModelConfig, gen: torch.Generator) -> dict:
    """The draws of inputs.make_weights, on the device.  One difference: the routed experts' output projections are
    scaled by 1 / sqrt(2 n_layers), the usual initialisation of projections into the residual stream.  The top-k choice
    of the router is a step function, so any change of rounding flips the near-ties among its logits; scaled so, a
    flipped choice moves its row by about two percent instead of ten and outputs can still be compared."""
    d, qd, kvd, dt = cfg.d_model, cfg.q_dim, cfg.kv_dim, cfg.torch_dtype

    def mat(*shape, std=0.02):
        return torch.empty(shape, dtype=dt, device="cuda").normal_(0.0, std, generator=gen)

    def vec(n, mean, std):
        return torch.empty(n, dtype=torch.float32, device="cuda").normal_(mean, std, generator=gen)

    w = {"embed_primary": mat(cfg.vocab, d), "embed_branch": mat((cfg.n_paths - 1) * cfg.vocab, d),
         "embed_norm_g": vec(d, 1.0, 0.02), "final_norm_g": vec(d, 1.0, 0.02), "lm_head": mat(cfg.vocab, d), "layers": []}
    for _ in range(cfg.n_layers):
        lw = {"attn_norm_g": vec(d, 1.0, 0.02), "wq": mat(qd, d), "wk": mat(kvd, d), "wv": mat(kvd, d), "wo": mat(d, qd),
              "coup_a": vec(qd, 0.0, 0.5), "mlp_norm_g": vec(d, 1.0, 0.02), "coup_c": vec(d, 0.0, 0.5)}
        if cfg.is_moe:
            E, Fe, Fs = cfg.n_experts, cfg.d_expert, cfg.n_shared_experts * cfg.d_expert
            lw.update(router=mat(E, d, std=d ** -0.5), exp_gate=mat(E, Fe, d), exp_up=mat(E, Fe, d), exp_down=mat(E, d, Fe, std=0.02 * (2 * cfg.n_layers) ** -0.5),
                      sh_gate=mat(Fs, d), sh_up=mat(Fs, d), sh_down=mat(d, Fs), coup_b=vec(Fs, 0.0, 0.5))
            if cfg.compute_matched:
                lw.update(gate_a=vec(d, 1.0, 0.5), gate_g=vec(d, 1.0, 0.5))
        else:
            F = cfg.d_ff
            lw.update(w_gate=mat(F, d), w_up=mat(F, d), w_down=mat(d, F), coup_b=vec(F, 0.0, 0.5))
        w["layers"].append(lw)
    return w


def prepare(case: dict, seed: int) -> dict:
    cfg, B = _config(case), case["batch"]
    prompt = case["kind"] == "prompt"
    new = case["ctx"] if prompt else case["steps"]
    lens = _cached_lengths(case)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    # pages that the pass writes stand together at the pool's end, so that they can be looked at in place; the pages
    # of the cached contexts are scattered
    fresh = (new + PAGE - 2) // PAGE + 1
    pages = max(lens) // PAGE + fresh
    model = binding.Model(cfg, _weights(cfg, gen), B, pages * PAGE)
    first_fresh = model.num_pages - B * fresh
    table = torch.empty(B, pages, dtype=torch.int32)
    host = torch.Generator().manual_seed(seed)
    old = torch.randperm(first_fresh, generator=host).to(torch.int32).view(B, pages - fresh)
    for b, n in enumerate(lens):
        at = n // PAGE
        table[b, :at] = old[b, :at]
        table[b, at:at + fresh] = torch.arange(fresh, dtype=torch.int32) + (first_fresh + b * fresh)
        table[b, at + fresh:] = old[b, at:]
    model.set_page_table(table)
    pool = model.kv_view()
    if max(lens) > 0:
        for layer in range(cfg.n_layers):
            pool[layer, 0].normal_(0.0, 1.0, generator=gen)
            pool[layer, 1].normal_(0.0, 0.9, generator=gen)
    written = pool[:, :, first_fresh:]
    # The next tokens are left out for mixtures of experts: they are the argmax of the logits returned beside them, and
    # a row whose router near-tie flips takes another one too often for a share of a few dozen tokens.
    state = {"model": model, "lens": torch.tensor(lens, dtype=torch.int32), "written": written, "prompt": prompt,
             "returned": ("z1", "z2", "logits", "alpha") + (() if cfg.is_moe else ("next",))}
    shape = (B, new) if prompt else (new, B)
    state["tokens"] = torch.randint(0, cfg.vocab, shape, generator=gen, dtype=torch.int32, device="cuda")
    if not prompt:
        paths = 1 if case.get("primary_only") else cfg.n_paths
        state["step"] = (torch.empty(B, dtype=torch.int32, device="cuda"), torch.empty(B, dtype=torch.int32, device="cuda"),
                         torch.empty(paths, B, cfg.vocab, device="cuda"), torch.empty(B, device="cuda"))
        state["kept"] = {"next": torch.empty(new, B, dtype=torch.int32, device="cuda"),
                         "logits": torch.empty(new, paths, B, cfg.vocab, device="cuda"),
                         "alpha": torch.empty(new, B, device="cuda")}
        if paths == 1:
            del state["kept"]["alpha"]
        state["primary_only"] = paths == 1
    return state


def run(state: dict):
    model = state["model"]
    if state["prompt"]:
        if int(state["lens"][0]) == 0:
            model.reset()
        else:
            model.set_seq_lens(state["lens"])
        out = model.prefill_boundary(state["tokens"])
        return {**{k: v for k, v in out.items() if k in state["returned"]}, "kv": state["written"]}
    model.set_seq_lens(state["lens"])
    token, nxt, logits, alpha = state["step"]
    kept = state["kept"]
    for t in range(state["tokens"].shape[0]):
        token.copy_(state["tokens"][t])
        if state["primary_only"]:
            model.decode_step_primary_only(token, nxt, logits[0])
        else:
            model.decode_step(token, nxt, logits[0], logits[1:], alpha)
            kept["alpha"][t].copy_(alpha)
        kept["next"][t].copy_(nxt)
        kept["logits"][t].copy_(logits)
    return {**{k: v for k, v in kept.items() if k in state["returned"]}, "kv": state["written"]}


def _layer_params(cfg: ModelConfig, experts: float, shared: bool = True) -> float:
    """Elements of one layer's matrices, with `experts` routed experts."""
    n = 2 * cfg.q_dim * cfg.d_model + 2 * cfg.kv_dim * cfg.d_model
    if not cfg.is_moe:
        return n + 3 * cfg.d_ff * cfg.d_model
    return n + cfg.n_experts * cfg.d_model + 3 * cfg.d_expert * cfg.d_model * (experts + (cfg.n_shared_experts if shared else 0))


def _experts_loaded(cfg: ModelConfig, rows: int, branch_rows: int) -> float:
    """Distinct experts that so many rows select, on average, when their choices are independent."""
    if not cfg.is_moe:
        return 0.0
    E = cfg.n_experts
    miss = (1 - cfg.k_primary / E) ** rows
    if not cfg.router_mode:
        miss *= (1 - cfg.k_branch / E) ** branch_rows
    return E * (1 - miss)


def _step_work(cfg: ModelConfig, B: int, keys: float, paths: int) -> tuple[float, float]:
    """Bytes and operations of one decode step that reads `keys` cached positions over all sequences."""
    loaded = _experts_loaded(cfg, B, (paths - 1) * B)
    eb = cfg.elem_bytes
    nbytes = (cfg.n_layers * _layer_params(cfg, loaded) + cfg.vocab * cfg.d_model) * eb
    nbytes += keys * cfg.kv_bytes_per_token() + B * cfg.kv_bytes_per_token() + 4 * paths * B * cfg.vocab
    attn_paths = 1 if cfg.compute_matched else paths
    flops = 2.0 * paths * B * cfg.vocab * cfg.d_model + 4.0 * cfg.q_dim * cfg.n_layers * keys * attn_paths
    kb = cfg.k_primary if cfg.router_mode else cfg.k_branch
    flops += 2.0 * B * cfg.n_layers * _layer_params(cfg, cfg.k_primary)
    branch = _layer_params(cfg, kb, shared=not cfg.compute_matched)
    branch -= 2 * cfg.kv_dim * cfg.d_model  # a branch forms no key or value
    if cfg.compute_matched:
        branch -= 2 * cfg.q_dim * cfg.d_model
    return nbytes, flops + 2.0 * (paths - 1) * B * cfg.n_layers * branch


def work(case: dict) -> dict:
    cfg, B, lens = _config(case), case["batch"], _cached_lengths(case)
    if case["kind"] == "decode":
        paths = 1 if case.get("primary_only") else cfg.n_paths
        nbytes = flops = 0.0
        for t in range(case["steps"]):
            b, f = _step_work(cfg, B, sum(lens) + B * (t + 1), paths)
            nbytes, flops = nbytes + b, flops + f
        return {"bytes": nbytes, "flops": flops}
    n, past = case["ctx"] - 1, lens[0]
    tokens = B * n
    pairs = B * (n * past + n * (n + 1) / 2.0)
    flops = 2.0 * tokens * cfg.n_layers * _layer_params(cfg, cfg.k_primary) + 4.0 * cfg.q_dim * cfg.n_layers * pairs
    # each matrix and the cached prefix read once for the whole call, the cache's new positions written once
    all_experts = _experts_loaded(cfg, tokens, B)
    b, f = _step_work(cfg, B, B * (past + n + 1), cfg.n_paths)
    nbytes = (cfg.n_layers * _layer_params(cfg, all_experts) + cfg.vocab * cfg.d_model) * cfg.elem_bytes
    nbytes += (B * past + tokens + B) * cfg.kv_bytes_per_token() + 4 * cfg.n_paths * B * cfg.vocab
    return {"bytes": nbytes, "flops": flops + f}


def tolerance(case: dict):
    """About four times what the library's own alternative chains (the generic CUDA-core kernels and attention, the
    16-row prompt attention) differ by from its default on the same inputs.  Largest relative errors seen, logits /
    cache: 4e-4 / 4e-4 in bf16 decode steps, 7e-4 / 1.8e-3 in prompts (K and V are rounded to bf16 after every layer,
    one unit in the last place being 7.8e-3 of a value); mixtures of experts 6e-4 / 2e-4 and 1.2e-3 / 3.2e-3, with
    single values off by 2e-2 and 1.9e-1 where a near-tie in the router fell the other way.  One such row among few
    weighs more, hence the second term."""
    if case["model"] == "tiny":
        return {"rel": 1e-5}
    prompt = case["kind"] == "prompt"
    if case["model"] == "moe":
        rows = case["batch"] * (1 if prompt else 2 * case["steps"])
        return {"rel": (1e-2 if prompt else 2.5e-3) + (0.02 if prompt else 0.03) * rows ** -0.5, "max": 0.8}
    return {"rel": 8e-3 if prompt else 2e-3, "max": 8e-2 if prompt else 5e-2}
