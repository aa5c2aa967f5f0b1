"""What a user of this library has it do, as measurable cases: draft steps, and the two calls that stand next to them.

Three kinds of work, each through the public entry points:

  step     one block-parallel draft step (`Drafter.draft`) over a batch of requests: token ids and logits
  verify   the draft probabilities of a block's tokens from its logits (`hspec_op_token_probs`), then the acceptance rule of
           speculative decoding (`hspec_op_accept`)
  lm_head  LM head and arg-max for hosts that cannot allocate while drafting (`hspec_op_lm_head_argmax_noalloc`)

Sizes are the drafter shapes this repository is configured for, over its range of concurrency (1 to 256 requests), block
length (1 to 32 positions) and context length.  Weights, target KV, hidden states and logits are seeded random draws with
the scales of the repository's workloads: matrices N(0, 0.02), K/V and hidden states N(0, 1).
"""
import math
import zlib

import torch

import paper_2609_24197_b200 as hs

# drafter shapes: an 8B-class and a 32B-class target, the paper's own drafter for an 8B-class target (five fused hidden
# states, small Mamba state, three attention layers of four, causal-correction head), and a test-sized one
SHAPES = {
    "8b": dict(D=4096, n_fuse=1, r=4096, L=2, has_attn=[1, 1], kv_slot=[0, 1], n_slots=2, Di=8192, P=64, N=128, G=4,
               d_conv=4, dt_rank=0, Hq=32, Hkv=8, dh=128, rope_theta=1.0e6, qk_norm=1, F=14336, V=128256, markov_rank=0),
    "32b": dict(D=5120, n_fuse=1, r=5120, L=2, has_attn=[1, 1], kv_slot=[0, 1], n_slots=2, Di=10240, P=64, N=128, G=4,
                d_conv=4, dt_rank=0, Hq=64, Hkv=8, dh=128, rope_theta=1.0e6, qk_norm=1, F=25600, V=152064, markov_rank=0),
    "paper_8b": dict(D=4096, n_fuse=5, r=4096, L=4, has_attn=[1, 1, 1, 0], kv_slot=[0, 1, 2, -1], n_slots=3, Di=3072, P=64,
                     N=4, G=4, d_conv=4, dt_rank=0, Hq=32, Hkv=8, dh=128, rope_theta=1.0e6, qk_norm=1, F=12288, V=151936,
                     markov_rank=256),
    "tiny": dict(D=256, n_fuse=1, r=256, L=1, has_attn=[1], kv_slot=[0], n_slots=1, Di=512, P=64, N=16, G=1, d_conv=4,
                 dt_rank=16, Hq=4, Hkv=2, dh=64, rope_theta=1.0e4, qk_norm=1, F=1024, V=1024, markov_rank=0),
}


def _step(name, shape, batch, block, ctx_low, ctx_high, spread="uniform", window=0, bf16=False, v_draft=0, markov=0):
    return dict(name=name, kind="step", shape=shape, batch=batch, block=block, ctx_low=ctx_low, ctx_high=ctx_high,
                spread=spread, window=window, bf16=bf16, v_draft=v_draft, markov=markov)


def listed():
    return [
        # smallest step: the test-sized drafter for one request; launches and host time are all there is
        _step("tiny_b1", "tiny", 1, 8, 256, 256),
        # one user waiting for tokens: weights are streamed for 16 rows
        _step("step_8b_b1", "8b", 1, 16, 2048, 2048),
        # a handful of requests of very different length and an odd block, as after uneven acceptance
        _step("step_8b_b5_ragged", "8b", 5, 7, 3, 16384, spread="log"),
        # ordinary serving batch
        _step("step_8b_b32", "8b", 32, 16, 512, 8192),
        # the same with bf16 operands (no library copy of the weights) and the paper's 2048-token window, a batch in between
        _step("step_8b_b61_bf16_window", "8b", 61, 9, 500, 12000, window=2048, bf16=True),
        # the paper's own drafter with its window and its rank-256 causal-correction head over the whole vocabulary
        _step("step_paper_b32", "paper_8b", 32, 8, 512, 8192, window=2048, markov=256),
        # high concurrency on a 32B-class target, long contexts
        _step("step_32b_b128", "32b", 128, 16, 1024, 32768, spread="log"),
        # the same target with the pruned 32 000-token drafter vocabulary and the causal-correction head the paper serves
        _step("step_32b_b96_pruned_markov", "32b", 96, 16, 1024, 32768, spread="log", v_draft=32000, markov=256),
        # the largest batch and block of the concurrency sweep
        _step("step_8b_b256_k32", "8b", 256, 32, 1024, 16384),
        # acceptance of one request's block, and of a full batch's
        dict(name="verify_b1", kind="verify", batch=1, block=16, vocab=128256),
        dict(name="verify_b128", kind="verify", batch=128, block=16, vocab=152064),
        # LM head of a host without an allocator: an odd number of rows
        dict(name="lm_head_m77", kind="lm_head", rows=77, width=5120, vocab=152064, bf16=False),
    ]


def _log_int(rng, low, high):
    return min(high, max(low, int(round(math.exp(rng.uniform(math.log(low), math.log(high + 0.49)))))))


def draw(rng):
    """One more case of the listed ranges (never costlier than the largest listed one)."""
    kind = rng.choice(["step", "step", "step", "step", "step", "verify", "lm_head"])
    if kind == "verify":
        return dict(kind="verify", batch=_log_int(rng, 1, 256), block=rng.randint(1, 32 if rng.random() < 0.3 else 16),
                    vocab=rng.choice([32000, 128256, 151936, 152064]))
    if kind == "lm_head":
        return dict(kind="lm_head", rows=_log_int(rng, 1, 512), width=rng.choice([4096, 5120]),
                    vocab=rng.choice([32000, 128256, 152064]), bf16=rng.random() < 0.5)
    shape = rng.choice(["8b", "8b", "8b", "32b", "paper_8b", "tiny"])
    top_batch, top_block, top_ctx = {"8b": (256, 32, 16384), "32b": (128, 16, 32768), "paper_8b": (128, 16, 16384),
                                     "tiny": (64, 32, 4096)}[shape]
    low = _log_int(rng, 1, 2048)
    case = _step(None, shape, _log_int(rng, 1, top_batch), rng.randint(1, top_block), low, _log_int(rng, low, top_ctx),
                 spread=rng.choice(["uniform", "log"]), window=rng.choice([0, 0, 2048]), bf16=rng.random() < 0.25)
    if shape == "32b":
        case["v_draft"] = rng.choice([0, 32000])
    if shape == "paper_8b" or (shape == "32b" and rng.random() < 0.3):
        case["markov"] = 256
    del case["name"]
    return case


# ------------------------------------------------------------------------------------------------ inputs

def _gen(seed, what):
    g = torch.Generator(device="cuda")
    g.manual_seed((int(seed) * 1000003 + zlib.crc32(what.encode())) % (1 << 62))
    return g


def _config(case):
    cfg = dict(SHAPES[case["shape"]], name=case["shape"], window=case["window"], rms_eps=1e-6, page_size=16,
               act_bf16=int(case["bf16"]), V_draft=case["v_draft"], markov_rank=case["markov"])
    cfg["mask_id"] = cfg["V"] - 1
    return cfg


def _sizes(cfg):
    heads = cfg["Di"] // cfg["P"]
    d_xbc = cfg["Di"] + 2 * cfg["G"] * cfg["N"]
    return dict(H=heads, d_S=heads * cfg["P"] * cfg["N"], d_xBC=d_xbc, d_in=cfg["Di"] + d_xbc + (cfg["dt_rank"] or heads),
                d_qkv=(cfg["Hq"] + 2 * cfg["Hkv"]) * cfg["dh"], Vd=cfg["V_draft"] or cfg["V"])


def _context_lengths(case):
    """The batch's context lengths, ascending: evenly spaced quantiles of the case's distribution, so that every seed has
    the same set (in another order)."""
    n, lo, hi = case["batch"], case["ctx_low"], case["ctx_high"]
    out = []
    for i in range(n):
        u = (i + 0.5) / n
        v = lo + u * (hi - lo) if case["spread"] == "uniform" else math.exp(math.log(lo) + u * (math.log(hi) - math.log(lo)))
        out.append(min(hi, max(lo, int(v))))
    return out


def _weights(cfg, seed):
    z = _sizes(cfg)
    D, F = cfg["D"], cfg["F"]

    def mat(name, *shape, std=0.02):
        return torch.empty(shape, dtype=torch.bfloat16, device="cuda").normal_(0.0, std, generator=_gen(seed, name))

    def vec(name, *shape, mean=0.0, std=0.02):
        return torch.empty(shape, dtype=torch.float32, device="cuda").normal_(mean, std, generator=_gen(seed, name))

    def uni(name, lo, hi, *shape):
        return torch.empty(shape, dtype=torch.float32, device="cuda").uniform_(lo, hi, generator=_gen(seed, name))

    w = {"embed": mat("embed", cfg["V"], D), "proj_r": mat("proj_r", cfg["r"], cfg["n_fuse"] * D),
         "proj_ds": mat("proj_ds", z["d_S"], cfg["r"]), "final_norm": vec("final_norm", D, mean=1.0),
         "lm_head": mat("lm_head", z["Vd"], D)}
    if cfg["V_draft"]:
        keep = torch.randperm(cfg["V"], generator=_gen(seed, "vocab_map"), device="cuda")[:cfg["V_draft"]]
        w["vocab_map"] = torch.sort(keep)[0].to(torch.int32)
    if cfg["markov_rank"]:
        # a trained bigram table is peaked: every token has a preferred successor, well above the rest (about 16 logits
        # against a spread of 1 in the table and 1.4 in the backbone's logits)
        r = cfg["markov_rank"]
        w["markov_in"] = mat("markov_in", cfg["V"], r, std=math.sqrt(16.0 / r))
        before = torch.randperm(z["Vd"], generator=_gen(seed, "successor"), device="cuda")
        tokens = w["vocab_map"].long()[before] if cfg["V_draft"] else before
        w["markov_out"] = w["markov_in"][tokens].contiguous()
    for l in range(cfg["L"]):
        p = f"layers.{l}."
        w[p + "mamba.norm"] = vec(p + "mamba.norm", D, mean=1.0)
        w[p + "mamba.in_proj"] = mat(p + "mamba.in_proj", z["d_in"], D)
        if cfg["dt_rank"]:
            w[p + "mamba.dt_up"] = mat(p + "mamba.dt_up", z["H"], cfg["dt_rank"])
        w[p + "mamba.conv_w"] = uni(p + "mamba.conv_w", -0.5, 0.5, z["d_xBC"], cfg["d_conv"])
        w[p + "mamba.conv_b"] = vec(p + "mamba.conv_b", z["d_xBC"])
        w[p + "mamba.A_log"] = uni(p + "mamba.A_log", 0.0, 2.0, z["H"])
        dt = torch.exp(uni(p + "mamba.dt_bias", math.log(1e-3), math.log(1e-1), z["H"]).double())
        w[p + "mamba.dt_bias"] = (dt + torch.log(-torch.expm1(-dt))).float()        # inverse softplus
        w[p + "mamba.Dskip"] = torch.ones(z["H"], device="cuda")
        w[p + "mamba.gnorm"] = vec(p + "mamba.gnorm", cfg["Di"], mean=1.0)
        w[p + "mamba.out_proj"] = mat(p + "mamba.out_proj", D, cfg["Di"])
        if cfg["has_attn"][l]:
            w[p + "attn.norm"] = vec(p + "attn.norm", D, mean=1.0)
            w[p + "attn.wqkv"] = mat(p + "attn.wqkv", z["d_qkv"], D)
            w[p + "attn.q_norm"] = vec(p + "attn.q_norm", cfg["dh"], mean=1.0)
            w[p + "attn.k_norm"] = vec(p + "attn.k_norm", cfg["dh"], mean=1.0)
            w[p + "attn.wo"] = mat(p + "attn.wo", D, cfg["Hq"] * cfg["dh"])
        w[p + "mlp.norm"] = vec(p + "mlp.norm", D, mean=1.0)
        w[p + "mlp.w_gate_up"] = mat(p + "mlp.w_gate_up", 2 * F, D)
        w[p + "mlp.w_down"] = mat(p + "mlp.w_down", D, F)
    return w


class _StepState:
    """A drafter with its weights loaded and one batch of requests over the target's paged KV cache."""

    def __init__(self, case, seed):
        cfg = _config(case)
        weights = _weights(cfg, seed)
        ctx = _context_lengths(case)
        order = torch.randperm(len(ctx), generator=_gen(seed, "order"), device="cuda").tolist()
        ctx = [ctx[i] for i in order]
        pages = [(c + 15) // 16 for c in ctx]
        perm = torch.randperm(max(1, sum(pages)), generator=_gen(seed, "pages"), device="cuda").to(torch.int32).cpu()
        table = torch.full((len(ctx), max(1, max(pages))), -1, dtype=torch.int32)
        at = 0
        for b, n in enumerate(pages):
            table[b, :n] = perm[at:at + n]
            at += n
        shape = (perm.numel(), 16, cfg["Hkv"], cfg["dh"])

        def pool(what):
            return torch.empty(shape, dtype=torch.bfloat16, device="cuda").normal_(generator=_gen(seed, what))

        tokens = torch.randint(0, cfg["V_draft"] or cfg["V"], (len(ctx),), generator=_gen(seed, "tokens"), device="cuda")
        if cfg["V_draft"]:
            tokens = weights["vocab_map"].long()[tokens]
        self.batch = dict(
            page_table=table.cuda(), ctx_lens=torch.tensor(ctx, dtype=torch.int32, device="cuda"),
            last_hidden=torch.empty((len(ctx), cfg["n_fuse"] * cfg["D"]), dtype=torch.bfloat16, device="cuda").normal_(
                generator=_gen(seed, "hidden")),
            last_token=tokens.to(torch.int32), k_pools=[pool(f"k{s}") for s in range(cfg["n_slots"])],
            v_pools=[pool(f"v{s}") for s in range(cfg["n_slots"])])
        self.block = case["block"]
        self.drafter = hs.Drafter(cfg, weights, max_batch=len(ctx), max_k=case["block"], max_ctx=max(1, max(ctx)))

    def __del__(self):
        if getattr(self, "drafter", None) is not None:
            torch.cuda.synchronize()
            self.drafter.close()


def prepare(case, seed):
    if case["kind"] == "step":
        return _StepState(case, seed)
    if case["kind"] == "verify":
        rows = case["batch"] * case["block"]
        logits = torch.empty((rows, case["vocab"]), dtype=torch.float32, device="cuda").normal_(0.0, 1.4, generator=_gen(seed, "logits"))
        ids = torch.argmax(logits, dim=1)
        # drafts are confident now and then: the chosen token leads by 0 to 12 logits
        lead = torch.empty(rows, device="cuda").uniform_(0.0, 12.0, generator=_gen(seed, "lead"))
        logits[torch.arange(rows, device="cuda"), ids] += lead
        p_target = torch.empty((case["batch"], case["block"]), device="cuda").uniform_(0.0, 1.0, generator=_gen(seed, "p"))
        alpha = torch.empty((case["batch"], case["block"]), device="cuda").uniform_(0.0, 1.0, generator=_gen(seed, "alpha"))
        return dict(case=case, logits=logits, ids=ids.to(torch.int32), p_target=p_target, alpha=alpha)
    kind = torch.bfloat16 if case["bf16"] else torch.float16
    x = torch.empty((case["rows"], case["width"]), dtype=kind, device="cuda").normal_(0.0, 1.0, generator=_gen(seed, "x"))
    w = torch.empty((case["vocab"], case["width"]), dtype=kind, device="cuda").normal_(0.0, 0.02, generator=_gen(seed, "w"))
    # the outputs are the caller's, laid out once: such a host cannot allocate here
    return dict(case=case, x=x, w=w, ids=torch.empty(case["rows"], dtype=torch.int32, device="cuda"),
                logits=torch.empty((case["rows"], case["vocab"]), dtype=torch.float32, device="cuda"))


def run(state):
    if isinstance(state, _StepState):
        ids, logits, _ = state.drafter.draft(state.batch, state.block, want_logits=True)
        return dict(ids=ids, logits=logits)
    case = state["case"]
    if case["kind"] == "verify":
        p_draft = torch.empty((case["batch"], case["block"]), dtype=torch.float32, device="cuda")
        n_accept = torch.empty(case["batch"], dtype=torch.int32, device="cuda")
        hs.hspec_op_token_probs(state["logits"], state["ids"], p_draft)
        hs.hspec_op_accept(state["p_target"], p_draft, state["alpha"], n_accept)
        return dict(p_draft=p_draft, n_accept=n_accept)
    hs.hspec_op_lm_head_argmax_noalloc(state["x"], state["w"], state["ids"], state["logits"])
    return dict(ids=state["ids"], logits=state["logits"])


# ------------------------------------------------------------------------------------------------ accounting

def work(case):
    if case["kind"] == "verify":
        rows = case["batch"] * case["block"]
        return {"bytes": 4.0 * rows * case["vocab"] + 20.0 * rows, "flops": 3.0 * rows * case["vocab"]}
    if case["kind"] == "lm_head":
        m, n, k = case["rows"], case["vocab"], case["width"]
        return {"bytes": 2.0 * n * k + 2.0 * m * k + 4.0 * m * n + 4.0 * m, "flops": 2.0 * m * n * k}
    cfg = _config(case)
    z = _sizes(cfg)
    D, F, L, B, k = cfg["D"], cfg["F"], cfg["L"], case["batch"], case["block"]
    M = B * k
    # a step's block rows are the last token's embedding and k - 1 times the mask's: before the first mixer there are no
    # more than B + 1 different rows
    mats = [(B, cfg["r"], cfg["n_fuse"] * D), (B, z["d_S"], cfg["r"]), (M, z["Vd"], D)]
    vectors, att, flops = D, 0.0, 0.0
    seen = [min(c, case["window"] - 1) if case["window"] else c for c in _context_lengths(case)]
    for l in range(L):
        mats += [(min(M, B + 1) if l == 0 else M, z["d_in"], D), (M, D, cfg["Di"]), (M, 2 * F, D), (M, D, F)]
        if cfg["dt_rank"]:
            mats.append((M, z["H"], cfg["dt_rank"]))
        vectors += 2 * D + cfg["Di"] + z["d_xBC"] * (cfg["d_conv"] + 1) + 3 * z["H"]
        flops += 4.0 * M * z["d_S"]
        if cfg["has_attn"][l]:
            mats += [(M, z["d_qkv"], D), (M, D, cfg["Hq"] * cfg["dh"])]
            vectors += D
            att += sum(seen) * cfg["Hkv"] * cfg["dh"] * 4.0
            flops += sum(4.0 * k * cfg["Hq"] * cfg["dh"] * (s + k / 2) for s in seen)
    if cfg["markov_rank"]:
        mats.append((M, z["Vd"], cfg["markov_rank"]))
    flops += sum(2.0 * m * n * kk for m, n, kk in mats)
    nbytes = sum(2.0 * n * kk for _, n, kk in mats) + 4.0 * vectors + att
    nbytes += 2.0 * B * cfg["n_fuse"] * D + 2.0 * (min(M, B + 1)) * D + 4.0 * M * z["Vd"] + 4.0 * M
    return {"bytes": nbytes, "flops": flops}


def tolerance(case):
    """About four times what the calls differ by from the same arithmetic in 64 bits (32 for the full-size steps): steps with
    fp16 operands rel 0.5e-3 to 1.4e-3 and 8e-3 at the largest, with bf16 operands 3.6e-3 to 7.4e-3 and 4e-2; the LM head
    (sums of 5120 products) 6e-6 and 4e-5; draft probabilities 2.2e-7 and 9e-7.  The arg-max of near-tied random logits
    moved on one or two of a hundred tokens."""
    if case["kind"] == "verify":
        return {"rel": 1e-6, "max": 4e-6, "differ": 0.02}
    if case["kind"] == "lm_head":
        return {"rel": 2.4e-5, "max": 1.6e-4, "differ": 0.02}
    tokens = case["batch"] * case["block"]
    differ = min(0.9, 0.05 + 3.0 / tokens)
    return {"rel": 3e-2, "max": 0.15, "differ": differ} if case["bf16"] else {"rel": 4e-3, "max": 3.5e-2, "differ": differ}
