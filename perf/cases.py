"""The work whose speed counts: decode steps and the prefill side (fit, encode) of one attention layer.

A case is one layer of one batch of sequences.  `prepare` builds what a serving process holds before the call (K/V caches,
packed codes, an installed or to-be-fitted projection, the step's inputs); `run` is one call of the library's public
entry points as a decode loop or a prefill makes it.  Shapes, head layouts, code lengths and budgets are those of the
package's own configurations (`inputs.CONFIGS`) and of the benchmark's latency sweep.
"""
from __future__ import annotations

import torch

from paper_2608_04405_b200 import binding as B
from paper_2608_04405_b200.inputs import Workload, WorkloadSpec

D = 128                      # head_dim of every configuration
ROOM = 256                   # decode steps a sequence may take before its slot starts over with the same prompt
RING = 4                     # distinct step inputs a decode loop cycles through
CAL_ROWS = 4096              # keys per unit the offline calibration looks at
MAX_KEYS = 32 * 131072       # keys of the largest listed prefill (batch 4 x 8 KV heads x 128K)


def _case(name, path, batch, heads, ctx, *, ctx_min=0, dtype="bf16", bits=128, ppm=20000, count=0, score="hamming", rope=500000.0):
    c = {"path": path, "batch": batch, "q_heads": heads[0], "kv_heads": heads[1], "ctx": ctx, "ctx_min": ctx_min, "dtype": dtype, "bits": bits,
         "ppm": ppm, "count": count, "score": score, "rope": rope}
    return dict(c, name=name) if name else c


# Head layouts (query heads, KV heads) of the configurations.
SINGLE, GQA4, GQA7 = (1, 1), (32, 8), (28, 4)


def listed():
    return [
        # decode: one token of one layer (cache write + sparse attention, the fused call)
        _case("step_4k_f32", "step", 1, SINGLE, 4096, dtype="f32", bits=64, rope=0.0),           # smallest call: latency only
        _case("step_32k", "step", 1, GQA4, 32768),                                               # one user, ordinary context
        _case("step_128k_b4", "step", 4, GQA4, 131072),                                          # the headline: long contexts, small batch
        _case("step_128k_b4_weighted", "step", 4, GQA4, 131072, score="weighted"),               # the paper's sign + magnitude score
        _case("step_128k_b8_g7", "step", 8, GQA7, 131072, rope=1000000.0),                       # odd number of query heads per KV head
        _case("step_ragged_b16", "step", 16, GQA4, 65536, ctx_min=16384),                        # a serving batch of unequal contexts
        _case("step_ragged_b16_256bit", "step", 16, GQA4, 65536, ctx_min=16384, bits=256),       # the same with the longest codes
        _case("step_1m_64bit", "step", 1, GQA4, 1048576, bits=64, ppm=0, count=2048),            # one very long context, fixed budget
        # prefill: the projection of every KV head from its own keys, then the codes of all cached keys
        _case("fit_32k", "fit", 1, GQA4, 32768),
        _case("fit_128k_b4", "fit", 4, GQA4, 131072),                                            # the largest
        _case("encode_128k_b4", "encode", 4, GQA4, 131072),
        _case("encode_4k_f32", "encode", 1, SINGLE, 4096, dtype="f32", bits=64, rope=0.0),
    ]


def _log_int(rng, lo, hi):
    return int(round(lo * (hi / lo) ** rng.random()))


def draw(rng):
    """Any path over the same ranges: contexts of 1K to 1M keys, batches of 1 to 16, 64 to 256 bits, every score option."""
    path = rng.choices(["step", "two_calls", "fit", "encode"], [60, 8, 16, 16])[0]
    if rng.random() < 0.1:                                   # fp32 caches: small single-head work
        return _case(None, path, _log_int(rng, 1, 4), SINGLE, _log_int(rng, 4096 if path == "fit" else 1024, 16384), dtype="f32", bits=rng.choice([64, 128]),
                     ppm=rng.choice([10000, 20000, 50000]), rope=0.0)
    heads = rng.choice([GQA4, GQA4, GQA7])
    bits = rng.choice([64, 128, 128, 256])
    batch = _log_int(rng, 1, 16)
    keys = MAX_KEYS if path in ("step", "two_calls") else MAX_KEYS * 128 // max(bits, 128)
    ctx = _log_int(rng, 4096 if path == "fit" else 1024, min(1048576, keys // (batch * heads[1])))
    score = rng.choices(["hamming", "weighted", "safeguard"], [70, 20, 10])[0] if path in ("step", "two_calls") else "hamming"
    if rng.random() < 0.25:
        ppm, count = 0, rng.choice([1024, 2048])             # fixed budgets
    else:
        ppm, count = rng.choice([10000, 20000, 50000]), 0
    ragged = batch > 1 and rng.random() < 0.5
    return _case(None, path, batch, heads, ctx, ctx_min=max(1, ctx // 4) if ragged else 0, bits=bits, ppm=ppm, count=count, score=score,
                 rope=500000.0 if heads == GQA4 else 1000000.0)


def _spec(case):
    return WorkloadSpec("case", 9, case["batch"], case["q_heads"], case["kv_heads"], case["ctx"], case["dtype"], case["bits"], case["ppm"], ROOM, 8,
                        rope_base=case["rope"] or None, n_ctx_min=case["ctx_min"] or None)


def _eas_ppm(case):
    """The safeguard set is a tenth of the budget, as the paper sizes it."""
    if case["score"] != "safeguard":
        return 0
    return max(1, case["ppm"] // 10 if case["ppm"] else case["count"] * 100000 // case["ctx"])


def _calibrate(k_cache, lens, v_star):
    """Offline calibration: Algorithm 1 on a sample of every unit's keys (a projection of the kind a fit leaves)."""
    batch, kv_heads = k_cache.shape[:2]
    rows = [k_cache[i][:, torch.arange(CAL_ROWS, device="cuda") * lens[i] // CAL_ROWS].float() for i in range(batch)]
    R = torch.cat(rows).view(batch * kv_heads, CAL_ROWS, D)
    P = torch.empty_like(v_star)
    for i in range(v_star.shape[1]):
        u = torch.where((R * v_star[:, i, None, :]).sum(-1) >= 0, 1.0, -1.0)
        P[:, i] = (u[..., None] * R).mean(1)
        R -= u[..., None] * P[:, i, None, :]
    return P


class _Layer:
    """One layer's caches, codes and context, and the inputs of the next decode steps."""

    def __init__(self, case, seed):
        self.path, self.spec = case["path"], _spec(case)
        s = self.spec
        w = Workload(s, device="cuda", extra_rows=ROOM, salt=seed)
        self.kv, self.k, self.v = B.interleaved_kv(s.batch, s.n_kv_heads, w.n_max, D, s.torch_dtype)
        self.k.copy_(w.k_cache)
        self.v.copy_(w.v_cache)
        self.lens, self.v_star = w.seq_lens, w.v_star
        self.budget = {"budget_ppm": case["ppm"], "budget_count": case["count"]}
        self.ctx = B.Context(B.make_config(s.batch, s.n_q_heads, s.n_kv_heads, w.n_max, s.code_bits, s.torch_dtype, kv_row_stride=2 * D,
                                           score_mode=B.BPC_SCORE_WEIGHTED7 if case["score"] == "weighted" else B.BPC_SCORE_HAMMING,
                                           eas_ppm=_eas_ppm(case)))
        self.ctx.set_seq_lens(self.lens)
        if self.path == "fit":
            self.workspace = torch.empty(self.ctx.fit_workspace_bytes(), dtype=torch.uint8, device="cuda")
            return
        self.codes = self.ctx.alloc_codes()
        self.ctx.set_projection(_calibrate(self.k, self.lens, self.v_star))
        if self.path == "encode":
            return
        self.ctx.encode_keys(self.k, self.codes)
        if case["score"] == "safeguard":
            self.ctx.build_eas()
        self.inputs = [(*w.new_kv(self.lens), w.queries(self.lens)[0]) for _ in range(RING)]
        self.steps = 0

    def next_inputs(self):
        if self.steps == ROOM:                               # the slot is full: the next request brings the same prompt
            self.ctx.set_seq_lens(self.lens)
            self.steps = 0
        self.steps += 1
        return self.inputs[self.steps % RING]

    def step(self):
        k_new, v_new, q = self.next_inputs()
        return self.ctx.append_decode_attn(k_new, v_new, self.k, self.v, self.codes, q, **self.budget)

    def two_calls(self):
        k_new, v_new, q = self.next_inputs()
        self.ctx.append(k_new, v_new, self.k, self.v, self.codes)
        return self.ctx.decode_attn(q, self.k, self.v, self.codes, **self.budget)


def prepare(case, seed):
    return _Layer(case, seed)


def run(state):
    if state.path == "fit":
        state.ctx.fit(state.k, state.v_star, state.workspace)
        return dict(zip(("P", "P_hash", "gram"), state.ctx.get_projection()))
    if state.path == "encode":
        state.ctx.encode_keys(state.k, state.codes)
        return {"codes": state.codes}
    out = state.step() if state.path == "step" else state.two_calls()
    return {"out": out, "codes": state.codes, "kv": state.kv}


def work(case):
    """Each input once and each result once.  Ragged lengths are drawn from the seed: their mean stands in."""
    n = (case["ctx"] + case["ctx_min"]) // 2 if case["ctx_min"] else case["ctx"]
    units, b, esz = case["batch"] * case["kv_heads"], case["bits"], 2 if case["dtype"] == "bf16" else 4
    group = case["q_heads"] // case["kv_heads"]
    if case["path"] == "fit":                                # keys and directions in; P, its rounding and the Gram matrix out
        return {"bytes": units * (n * D * esz + 3 * b * D * 4 + b * b * 4), "flops": units * 4 * n * b * D}
    if case["path"] == "encode":                             # keys and projection in, codes out; GEMM and greedy sweep
        return {"bytes": units * (n * D * esz + b * D * esz + n * b // 8), "flops": units * n * (2 * b * D + b * b)}
    k = min(n, case["count"] or -(-n * case["ppm"] // 1000000))
    step = n * b // 8 + 2 * k * D * esz + group * D * (esz + 4) + 4 * D * esz + b * D * esz
    return {"bytes": units * step, "flops": units * group * (4 * k * D + 2 * b * D)}


def tolerance(case):
    """What the data types leave open between two correct implementations."""
    if case["path"] == "fit":
        # A decision inside the fp32 rounding band may come out either way, and Algorithm 1 carries that one sign on into
        # every later bit; one key of n weighs 1/n.  Between the library's two passes (tensor cores, CUDA cores): up to
        # 6e-3 at 4K keys, 2e-3 at 32K and 6e-4 at 128K.
        rel = 0.03 * min(1.0, (2048 / (case["ctx_min"] or case["ctx"])) ** 0.5)
        return {"rel": rel, "max": 25 * rel}
    if case["path"] == "encode":
        return {"rel": 0.0, "differ": 1e-4}                  # bits whose decision value is zero to fp32 rounding
    # selection is exact on equal codes; the attention sums are fp32 (bf16 caches) or fp64
    return {"rel": 1e-3 if case["dtype"] == "bf16" else 1e-5, "max": 2e-2 if case["dtype"] == "bf16" else 1e-3, "differ": 1e-4}
