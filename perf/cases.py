"""Performance cases of the bidirectional Mamba mixer and its layer stacks: what programs that use this library call, over
the sizes they call it with.

Every case goes through the public entry points of `paper_2511_15927_b200.binding`.  Sizes are those of the configurations in
`inputs.CONFIGS` and `bench.py` (d_model 128 to 2048, the paper's 1.3B widths, vocabulary 50304) and ragged ones between them.
Stack cases return the logits and do not ask for the arg-max: with random weights the two largest of 50304 logits are often
within the rounding of bf16, so that the ids say nothing about the arithmetic.

    listed()          the named cases
    draw(rng)         one more case of the same kinds and ranges
    prepare(case, s)  inputs, weights and workspace on the GPU, from the seed
    run(state)        one call, as a user's program makes it
    work(case)        bytes and operations of one call that no implementation can avoid
    tolerance(case)   how far two correct implementations may be apart
"""
import math

import torch

from paper_2511_15927_b200 import binding as dm

VOCAB = 50304          # rows of the embedding and of the vocabulary projection
VOCAB_REAL = 50257     # ids that occur; the next one is the mask
MASK_ID = 50257
K = 4                  # taps of the depthwise conv
EXPAND = 2
NORM_EPS = 1e-5
ATTN_PERIOD = 5        # the hybrid: an attention mixer in layers 0, 5, 10, ...
D_COND = 128           # width of the timestep embedding

# (d_model, heads, d_state) of the models in the configurations: 64 x 64 heads, the 24-layer stack, its wide-state reading and the
# paper's 1.3B model (120 heads of 32)
WIDE, STACK, STACK_N128, PAPER = (2048, 64, 128), (1024, 32, 16), (1024, 32, 128), (1920, 120, 128)


def _case(name, kind, dtype, batch, seqlen, model, layers=1, prefix=0, commit=False):
    c = {"kind": kind, "dtype": dtype, "batch": batch, "seqlen": seqlen, "d_model": model[0], "heads": model[1], "d_state": model[2],
         "layers": layers, "prefix": prefix, "commit": commit}
    return dict(c, name=name) if name else c


def listed():
    return [
        # the smallest call: one fp32 layer on one short sequence (parity runs, small models): launches and latency
        _case("mixer_f32_256", "mixer", "f32", 1, 256, (128, 8, 16)),
        # one layer of the paper's model on one short sequence: the latency of a single request
        _case("mixer_paper_1k", "mixer", "bf16", 1, 1024, PAPER),
        # a batch whose length is no multiple of any tile
        _case("mixer_ragged", "mixer", "bf16", 3, 1111, STACK_N128),
        # the ordinary throughput point of one layer
        _case("mixer_batch", "mixer", "bf16", 8, 2048, WIDE),
        # one long sequence: few independent scans, each of them long
        _case("mixer_32k", "mixer", "bf16", 1, 32768, WIDE),
        # the throughput point from and to pinned host memory, copies included
        _case("host_batch", "mixer_host", "bf16", 8, 2048, WIDE),
        # block-autoregressive decoding, one layer: a 32-token block from a carried state, the new state committed
        _case("block_commit", "block", "bf16", 16, 32, WIDE, commit=True),
        # a denoising pass over the active block of 16 sequences through the whole stack (8 of 9 passes do not commit)
        _case("decode_b16", "decode", "bf16", 16, 32, WIDE, layers=24),
        # the paper's hybrid decoding one sequence: carried states and an 8192-token key/value cache, bound by reading the weights
        _case("decode_hybrid_b1", "decode_hybrid", "bf16", 1, 32, PAPER, layers=24, prefix=8192),
        # a full denoising step of the 24-layer stack
        _case("stack_4k", "stack", "bf16", 4, 4096, STACK, layers=24),
        # the paper's 1.3B model: timestep-conditioned blocks (AdaLN, mixer, AdaLN, MLP) at its batch-8 point
        _case("stack_cond_1k", "stack_cond", "bf16", 8, 1024, PAPER, layers=24),
        # the hybrid stack: full attention in every fifth layer, heads of 64
        _case("stack_hybrid_4k", "stack_hybrid", "bf16", 4, 4096, STACK, layers=24),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["mixer", "mixer", "mixer", "mixer_f32", "mixer_host", "block", "decode", "decode_hybrid", "stack", "stack_cond", "stack_hybrid"])
    if kind == "mixer":
        t = _log_int(rng, 80, 32768)
        b = rng.choice([1, 1, 2, 3, 4, 8])
        return _case(None, "mixer", "bf16", b, max(65, t // b), rng.choice([WIDE, STACK, STACK_N128, PAPER]))
    if kind == "mixer_f32":
        d = rng.choice([128, 192, 256])
        return _case(None, "mixer", "f32", rng.randint(1, 2), _log_int(rng, 48, 512), (d, d // 16, 16))
    if kind == "mixer_host":
        return _case(None, "mixer_host", "bf16", rng.randint(2, 8), _log_int(rng, 700, 2048), rng.choice([WIDE, PAPER]))
    if kind == "block":
        return _case(None, "block", "bf16", _log_int(rng, 1, 24), rng.randint(16, 64), rng.choice([WIDE, PAPER]), commit=rng.random() < 0.5)
    if kind == "decode":
        return _case(None, "decode", "bf16", _log_int(rng, 1, 16), rng.randint(16, 32), rng.choice([WIDE, PAPER, STACK]), layers=rng.randint(12, 24), commit=rng.random() < 0.2)
    if kind == "decode_hybrid":
        return _case(None, "decode_hybrid", "bf16", rng.randint(1, 4), rng.randint(16, 32), rng.choice([PAPER, STACK_N128]), layers=rng.randint(11, 24), prefix=_log_int(rng, 500, 8192))
    if kind == "stack":
        return _case(None, "stack", "bf16", rng.randint(1, 4), _log_int(rng, 300, 4096), rng.choice([STACK, STACK_N128]), layers=rng.randint(8, 24))
    if kind == "stack_cond":
        return _case(None, "stack_cond", "bf16", rng.randint(1, 8), _log_int(rng, 250, 1024), rng.choice([PAPER, STACK]), layers=rng.randint(6, 24))
    return _case(None, "stack_hybrid", "bf16", rng.randint(1, 4), _log_int(rng, 400, 4096), rng.choice([STACK, STACK_N128]), layers=rng.randint(6, 24))


# ------------------------------------------------------------------------------------------------ sizes

def _dims(case):
    d, h, n = case["d_model"], case["heads"], case["d_state"]
    di = EXPAND * d
    return {"d": d, "h": h, "n": n, "di": di, "p": di // h, "conv": di + 2 * n, "din": 2 * di + 2 * n + h, "t": case["batch"] * case["seqlen"],
            "attn_heads": d // (80 if d % 80 == 0 else 64)}


def _attn_layers(case):
    return [i for i in range(case["layers"]) if i % ATTN_PERIOD == 0] if "hybrid" in case["kind"] else []


def work(case):
    m, es = _dims(case), 2 if case["dtype"] == "bf16" else 4
    t, d, di, n, h = m["t"], m["d"], m["di"], m["n"], m["h"]
    n_attn = len(_attn_layers(case))
    n_mamba = case["layers"] - n_attn
    # one Mamba layer: both directions' projections, conv, recurrence (decay, outer product, contraction: 5 operations per state) and gate
    w_mamba = 2 * (m["din"] * d + di * d + (K + 1) * m["conv"] + di) * es + 2 * 3 * h * 4
    f_mamba = 2 * (2 * t * d * m["din"] + 2 * t * di * d + t * (2 * K * m["conv"] + 5 * di * n + 4 * di))
    state = case["batch"] * (di * n * 4 + (K - 1) * m["conv"] * es)            # one layer's carried state
    bytes_, flops = n_mamba * w_mamba, n_mamba * f_mamba
    if n_attn:
        keys = case["prefix"] + case["seqlen"]
        bytes_ += n_attn * (4 * d * d * es + 2 * case["batch"] * case["prefix"] * d * es)
        flops += n_attn * (8 * t * d * d + 4 * t * keys * d)
    if case["kind"] in ("block", "decode", "decode_hybrid"):
        bytes_ += n_mamba * state * (2 if case["commit"] else 1)
    if case["kind"] in ("mixer", "mixer_host", "block"):
        bytes_ += 2 * t * d * es
    else:
        bytes_ += t * 4 + min(t, VOCAB) * d * es + VOCAB * d * es + t * VOCAB * es
        flops += 2 * t * VOCAB * d
    if case["kind"] == "stack_cond":
        bytes_ += case["layers"] * (6 * d * D_COND + 2 * d * 2 * d) * es
        flops += case["layers"] * (8 * t * d * d + 12 * case["batch"] * d * D_COND)
    return {"bytes": float(bytes_), "flops": float(flops)}


def tolerance(case):
    # About four times what the same path shows against itself with its sums in another order: bf16, 32-token chunks of the scan in
    # place of 128-token ones: rel 1.2e-3, max 8.9e-3 for one layer and rel 1.4e-2, max 8.7e-2 through 24 layers (where rel stays
    # at twice that); fp32 against 64-bit sums: rel 5.5e-7, max 3.6e-6, times ten because that path has few roundings to begin with.
    if case["dtype"] == "f32":
        return {"rel": 5e-6, "max": 4e-5}
    if case["layers"] == 1:
        return {"rel": 5e-3, "max": 4e-2}
    return {"rel": 3e-2, "max": 3e-1}


# ------------------------------------------------------------------------------------------------ inputs

class _Draw:
    """Tensors on the GPU from one seed, with the distributions of inputs.py."""

    def __init__(self, seed, dtype):
        self.g = torch.Generator(device="cuda").manual_seed(seed)
        self.dt = torch.bfloat16 if dtype == "bf16" else torch.float32

    def normal(self, *sz, std=0.02, dtype=None):
        return torch.empty(*sz, device="cuda", dtype=dtype or self.dt).normal_(0.0, std, generator=self.g)

    def uniform(self, lo, hi, *sz, dtype=torch.float32):
        return torch.empty(*sz, device="cuda", dtype=torch.float32).uniform_(lo, hi, generator=self.g).to(dtype)

    def direction(self, m):
        dt = torch.exp(self.uniform(math.log(1e-3), math.log(1e-1), m["h"]))
        b = K ** -0.5
        return {"w_in": self.normal(m["din"], m["d"]), "conv_w": self.uniform(-b, b, m["conv"], K, dtype=self.dt),
                "conv_b": self.uniform(-b, b, m["conv"], dtype=self.dt), "A_log": torch.log(self.uniform(1.0, 16.0, m["h"])),
                "dt_bias": dt + torch.log(-torch.expm1(-dt)), "D": self.uniform(0.5, 1.5, m["h"]),
                "norm_w": self.uniform(0.5, 1.5, m["di"], dtype=self.dt), "w_out": self.normal(m["d"], m["di"])}

    def block(self, m):
        d = m["d"]
        base = torch.tensor([0.0, 1.0, 1.0], device="cuda").repeat_interleave(d).repeat(2)          # shift 0, scale 1, gate 1
        return {"w_cond": self.normal(6 * d, D_COND), "b_cond": base + self.normal(6 * d, std=0.1, dtype=torch.float32),
                "w_up": self.normal(2 * d, d), "b_up": self.normal(2 * d, dtype=torch.float32),
                "w_down": self.normal(d, 2 * d), "b_down": self.normal(d, dtype=torch.float32)}

    def tokens(self, b, length):
        ids = torch.randint(0, VOCAB_REAL, (b, length), generator=self.g, device="cuda", dtype=torch.int32)
        masked = self.uniform(0.0, 1.0, b, length) < self.uniform(0.0, 1.0, b, 1)                   # the forward masking process
        return torch.where(masked, torch.full_like(ids, MASK_ID), ids)


class _State:
    pass


def prepare(case, seed):
    m, r = _dims(case), _Draw(seed, case["dtype"])
    kind, b, length = case["kind"], case["batch"], case["seqlen"]
    s = _State()
    s.case, s.kind = case, kind
    s.cfg = dm.make_mixer_cfg(b, length, m["d"], EXPAND, m["n"], K, m["h"], dm.DM_BF16 if case["dtype"] == "bf16" else dm.DM_F32, norm_eps=NORM_EPS)
    s.stream = torch.cuda.current_stream().cuda_stream
    carried = kind in ("block", "decode", "decode_hybrid")
    attn = _attn_layers(case)
    if carried:                                     # the committed prefix of every layer, and where a commit goes
        s.ssm_in = r.normal(case["layers"], b, m["h"], m["p"], m["n"], std=0.5, dtype=torch.float32)
        s.conv_in = r.normal(case["layers"], b, K - 1, m["conv"], std=1.0)
        s.ssm_out = torch.zeros_like(s.ssm_in) if case["commit"] else None
        s.conv_out = torch.zeros_like(s.conv_in) if case["commit"] else None
    if kind in ("mixer", "mixer_host", "block"):
        s.keep = (r.direction(m), r.direction(m))
        s.w = tuple(dm.make_dir_weights(q) for q in s.keep)
        s.x = r.normal(b, length, m["d"], std=1.0)
        s.y = torch.zeros_like(s.x)
        nbytes = dm.dm_bimamba_workspace_bytes(s.cfg)
        if kind == "mixer_host":
            nbytes += 2 * ((s.x.numel() * s.x.element_size() + 255) // 256 * 256)
            s.x, s.y = s.x.cpu().pin_memory(), s.y.cpu().pin_memory()
    else:
        layers = [{"norm_w": r.uniform(0.5, 1.5, m["d"], dtype=r.dt), "fwd": r.direction(m), "rev": r.direction(m)} for _ in range(case["layers"])]
        s.keep = {"embed": r.normal(VOCAB, m["d"]), "w_vocab": r.normal(VOCAB, m["d"]), "final_norm_w": r.uniform(0.5, 1.5, m["d"], dtype=r.dt), "layers": layers}
        s.weights, s.keep_layers = dm.make_stack_weights(s.keep)
        s.cfg = dm.dm_stack_cfg(s.cfg, case["layers"], VOCAB, 1e-5)
        s.tokens = r.tokens(b, length)
        s.logits = torch.zeros(b, length, VOCAB, device="cuda", dtype=r.dt)
        if carried:
            s.states = (dm.dm_layer_state * case["layers"])()
            for i in range(case["layers"]):
                s.states[i] = dm.dm_layer_state(s.ssm_in[i].data_ptr(), s.conv_in[i].data_ptr(),
                                                s.ssm_out[i].data_ptr() if case["commit"] else None, s.conv_out[i].data_ptr() if case["commit"] else None)
        if attn:
            s.keep_attn = [{"w_qkv": r.normal(3 * m["d"], m["d"], std=m["d"] ** -0.5), "w_o": r.normal(m["d"], m["d"], std=0.5 * m["d"] ** -0.5)} if i in attn else None
                           for i in range(case["layers"])]
            s.attn_weights = dm.make_attn_weights(s.keep_attn)
            s.hybrid = dm.dm_hybrid_cfg(ATTN_PERIOD, m["attn_heads"])
        if kind == "decode_hybrid":
            cap = case["prefix"] + length
            s.k_cache = r.normal(len(attn), b, cap, m["d"], std=1.0)
            s.v_cache = r.normal(len(attn), b, cap, m["d"], std=1.0)
            s.attn_states = (dm.dm_attn_state * case["layers"])()
            for j, i in enumerate(attn):
                s.attn_states[i] = dm.dm_attn_state(s.k_cache[j].data_ptr(), s.v_cache[j].data_ptr(), case["prefix"], cap)
        if kind == "stack_cond":
            s.keep_blocks = [r.block(m) for _ in range(case["layers"])]
            s.block_weights = dm.make_block_weights(s.keep_blocks)
            s.block = dm.dm_block_cfg(2 * m["d"], D_COND, 1e-5)
            s.tau = r.normal(b, D_COND, std=1.0, dtype=torch.float32)
            nbytes = dm.dm_denoise_cond_workspace_bytes(s.cfg, s.block)
        elif attn:
            nbytes = dm.dm_denoise_hybrid_workspace_bytes(s.cfg)
        else:
            nbytes = dm.dm_denoise_workspace_bytes(s.cfg)
    s.workspace = torch.empty(nbytes, dtype=torch.uint8, device="cuda")
    return s


# ------------------------------------------------------------------------------------------------ one call

def run(s):
    ws, nb, kind = s.workspace.data_ptr(), s.workspace.numel(), s.kind
    if kind == "mixer":
        dm.dm_bimamba_forward(s.cfg, s.w, s.x.data_ptr(), s.y.data_ptr(), ws, nb, s.stream)
        return s.y
    if kind == "mixer_host":
        dm.dm_bimamba_forward_host(s.cfg, s.w, s.x.data_ptr(), s.y.data_ptr(), ws, nb, s.stream)
        return s.y
    if kind == "block":
        commit = s.ssm_out is not None
        dm.dm_bimamba_block_step(s.cfg, s.w, s.x.data_ptr(), s.ssm_in.data_ptr(), s.conv_in.data_ptr(), s.ssm_out.data_ptr() if commit else 0,
                                 s.conv_out.data_ptr() if commit else 0, s.y.data_ptr(), ws, nb, s.stream)
        return (s.y, s.ssm_out, s.conv_out) if commit else s.y
    if kind == "decode":
        dm.dm_denoise_step(s.cfg, s.weights, s.tokens.data_ptr(), s.logits.data_ptr(), 0, s.states, ws, nb, s.stream)
        return (s.logits, s.ssm_out, s.conv_out) if s.ssm_out is not None else s.logits
    if kind == "decode_hybrid":
        dm.dm_denoise_step_hybrid_block(s.cfg, None, s.hybrid, s.weights, None, s.attn_weights, s.tokens.data_ptr(), 0, s.logits.data_ptr(), 0,
                                        s.states, s.attn_states, ws, nb, s.stream)
        return s.logits, s.k_cache, s.v_cache
    if kind == "stack_cond":
        dm.dm_denoise_step_cond(s.cfg, s.block, s.weights, s.block_weights, s.tokens.data_ptr(), s.tau.data_ptr(), s.logits.data_ptr(), 0, None, ws, nb, s.stream)
        return s.logits
    if kind == "stack_hybrid":
        dm.dm_denoise_step_hybrid(s.cfg, None, s.hybrid, s.weights, None, s.attn_weights, s.tokens.data_ptr(), 0, s.logits.data_ptr(), 0, ws, nb, s.stream)
        return s.logits
    dm.dm_denoise_step(s.cfg, s.weights, s.tokens.data_ptr(), s.logits.data_ptr(), 0, None, ws, nb, s.stream)
    return s.logits
