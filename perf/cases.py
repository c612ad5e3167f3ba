"""The calls whose speed this library is about: what a serving program does with it, over the range it does it in.

Every case goes through the public entry points of ``paper_2510_12966_b200.binding`` on seeded synthetic logits of
``workloads`` (the generators of the tests and the benchmark). A case is a dict of plain values:

  path    "stage" (one model pair), "pyramid" (both stages in one call), "host" (the pyramid on host buffers) or
          "lmhead" (one stage whose large logits are produced inside the call by the LM-head GEMM)
  rows    whether the caller takes the per-row outputs (divergences, residual masses, token probabilities, window)
          besides the accept lengths and tokens; such calls use the ``_ex`` entry points

The integer results of a call sit in one [4, B] (or [2, B]) buffer that the program keeps and would copy to the
host as one piece.
"""
import math

import torch

from paper_2510_12966_b200 import binding, workloads

MODES = {"fuzzy": binding.FUZZY, "strict": binding.STRICT, "fallback": binding.FUZZY_SD_FALLBACK,
         "assisted": binding.ASSISTED}
DIVS = {"js": binding.DIV_JS, "tv": binding.DIV_TV, "kl": binding.DIV_KL}
# Noise of the drawn cases (sigma_q, sigma_d), and thresholds (stage 1, stage 2) in the middle of the divergences that
# it gives, so that both outcomes occur.
NOISE = {(0.7, 1.5): {"js": (0.25, 0.06), "tv": (0.55, 0.27), "kl": (1.3, 0.24)},
         (0.5, 2.0): {"js": (0.3, 0.03), "tv": (0.62, 0.19), "kl": (2.1, 0.12)},
         (0.3, 0.8): {"js": (0.08, 0.011), "tv": (0.33, 0.12), "kl": (0.36, 0.045)}}

# No drawn case reads more than the largest listed one (large_vocab), nor has a GEMM above that of the listed LM head.
MOST_BYTES = 256 * 20 * 152064 * 2
MOST_FLOPS = 2 * 256 * 4096 * 128256


def _case(path, B, K_d, K_q, V, dtype, **more):
    c = {"path": path, "B": B, "K_d": K_d, "K_q": K_q, "V": V, "dtype": dtype, "mode_q": "fuzzy", "mode_t": "fuzzy",
         "div": "js", "tau_q": 0.4, "tau_t": 0.2, "boost_lo": 8.0, "boost_hi": 8.0, "sigma_q": 0.7, "sigma_d": 1.5,
         "inv_temperature": 0.0, "bonus": False, "ragged": False, "rows": False, "d_model": 0}
    c.update(more)
    return c


def listed():
    named = {
        # The smallest call: one sequence, four fp32 positions of a 32000-token vocabulary, standard SD acceptance.
        # Launches and the host's part of the call are all of it.
        "stage_tiny": _case("stage", 1, 4, 4, 32000, "f32", mode_q="strict", tau_q=0.3, sigma_d=1.0),
        # Interactive decoding: one sequence through the whole pyramid at a 128256-token vocabulary, with the target's
        # own next token after an accepted window.
        "single_stream": _case("pyramid", 1, 8, 4, 128256, "bf16", bonus=True),
        # A few sequences with long windows: the assisted qualifier stage (a draw from the qualifier on rejection),
        # temperature 0.7, the target's bonus token, every per-row output taken (threshold tuning, logging).
        "assisted_bonus": _case("pyramid", 8, 20, 15, 128256, "bf16", mode_q="assisted", bonus=True, rows=True,
                                inv_temperature=1.0 / 0.7),
        # Batched serving, acceptance varying over the batch: the benchmark's workload.
        "serving": _case("pyramid", 64, 16, 8, 128256, "bf16", boost_lo=4.0, boost_hi=12.0),
        # The largest call: a big batch on a large vocabulary, low acceptance, so that most sequences draw.
        "large_vocab": _case("pyramid", 256, 8, 4, 152064, "bf16", tau_q=0.2, sigma_q=0.5, sigma_d=2.0),
        # fp32 logits (engines that keep them), half the batch for the same bytes.
        "large_vocab_f32": _case("pyramid", 128, 8, 4, 152064, "f32", tau_q=0.2, sigma_q=0.5, sigma_d=2.0),
        # A vocabulary of odd size: rows start at any 2-byte boundary.
        "odd_vocab": _case("pyramid", 32, 8, 4, 50257, "bf16"),
        # Batched serving with the KL divergence as the fuzzy criterion.
        "serving_kl": _case("pyramid", 64, 16, 8, 128256, "bf16", div="kl", tau_q=2.0, tau_t=1.0, boost_lo=4.0,
                            boost_hi=12.0),
        # One stage on windows of different lengths, standard SD acceptance, per-row outputs.
        "stage_ragged": _case("stage", 48, 16, 16, 32000, "f32", mode_q="strict", ragged=True, rows=True, sigma_d=1.0),
        # LM head fused into the target stage: a batch of 256 positions.
        "lmhead": _case("lmhead", 32, 8, 8, 128256, "bf16", tau_q=0.2, d_model=4096, rows=True),
        # The same for a handful of sequences, where streaming the weight is all of it.
        "lmhead_small": _case("lmhead", 3, 5, 5, 32000, "bf16", tau_q=0.2, d_model=2048, rows=True),
        # Logits in (pinned) host memory: the copies are part of the call.
        "host_batch": _case("host", 4, 8, 4, 128256, "bf16", mode_q="strict", mode_t="strict"),
    }
    return [dict(c, name=n) for n, c in named.items()]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _vocab(rng):
    V = _log_int(rng, 4000, 152064)
    kind = rng.random()
    if kind < 0.15:
        return V | 1                      # odd: no row but the first is aligned
    if kind < 0.25:
        return V // 2 * 2
    return max(V // 64 * 64, 4032)        # what padded vocabularies look like


def draw(rng):
    path = rng.choices(["stage", "pyramid", "lmhead", "host"], [3, 8, 2, 1])[0]
    V = _vocab(rng)
    dtype = "f32" if rng.random() < 0.3 else "bf16"
    K_d = rng.randint(1, 32) if rng.random() < 0.3 else rng.randint(3, 16)
    boost = rng.choice([(8.0, 8.0), (4.0, 12.0), (0.0, 4.0)])
    noise = rng.choice(sorted(NOISE))
    common = dict(boost_lo=boost[0], boost_hi=boost[1], sigma_q=noise[0], sigma_d=noise[1])
    if path == "lmhead":
        d_model = 64 * rng.randint(8, 64)
        B = _log_int(rng, 1, 48)
        K_d = rng.randint(2, 10)
        while 2 * B * K_d * d_model * V > MOST_FLOPS:
            B = (B + 1) // 2
        return _case("lmhead", B, K_d, K_d, V, "bf16", mode_q=rng.choice(["fuzzy", "fuzzy", "strict"]), tau_q=0.05,
                     d_model=d_model, rows=B < 8 or rng.random() < 0.5, **common)
    div = rng.choices(["js", "kl", "tv"], [8, 2, 1])[0] if path == "pyramid" else "js"
    tau = NOISE[noise][div]
    B = rng.randint(1, 8) if path == "host" else _log_int(rng, 1, 256)
    if path == "stage":
        K_q = K_d
    else:
        K_q = rng.randint(1, K_d)
    size = 4 if dtype == "f32" else 2
    while B * 3 * K_d * V * size > MOST_BYTES:
        B = (B + 1) // 2
    mode_q = rng.choice(["fuzzy", "fuzzy", "fuzzy", "strict", "assisted", "fallback"])
    if path == "host":
        mode_q = "strict"
    mode_t = mode_q if path == "host" or (mode_q != "assisted" and rng.random() < 0.7) else "fuzzy"
    return _case(path, B, K_d, K_q, V, dtype, mode_q=mode_q, mode_t=mode_t, div=div, tau_q=tau[0], tau_t=tau[1],
                 inv_temperature=rng.choice([0.0, 0.0, 1.0 / 0.7]) if path != "host" else 0.0,
                 bonus=path == "pyramid" and K_q < K_d and rng.random() < 0.15,
                 ragged=path == "stage" and rng.random() < 0.5,
                 rows=path != "host" and (B < 8 or rng.random() < 0.4), **common)


def prepare(case, seed):
    dev = torch.device("cuda")
    binding.load_library()
    binding.set_stream()
    B, K_d, K_q, V = case["B"], case["K_d"], case["K_q"], case["V"]
    boost = (case["boost_lo"], case["boost_hi"])
    state = {"case": case, "seed": seed % (1 << 31)}
    if case["path"] == "lmhead":
        state["inputs"] = workloads.make_fused_inputs(B, K_d, V, case["d_model"], seed, case["sigma_q"], device=dev)
        return state
    if case["path"] == "stage":
        state["inputs"] = workloads.make_stage_inputs(B, K_d, V, case["dtype"], seed, boost, case["sigma_d"], device=dev)
        if case["ragged"]:
            g = torch.Generator(device=dev)
            g.manual_seed(seed + 1)
            state["n_valid"] = torch.randint(0, K_d + 1, (B,), generator=g, device=dev, dtype=torch.int32)
        state["results"] = torch.empty((2, B), dtype=torch.int32, device=dev)
        state["out"] = tuple(state["results"])
        return state
    inputs = workloads.make_pyramid_inputs(B, K_d, K_q + (1 if case["bonus"] else 0), V, case["dtype"], seed, boost,
                                           case["sigma_q"], case["sigma_d"], device=dev)
    results = torch.empty((4, B), dtype=torch.int32, device=dev)
    if case["path"] == "host":
        inputs = [t.cpu().pin_memory() for t in inputs]
        results = results.cpu().pin_memory()
    state["inputs"] = inputs
    state["results"] = results
    state["out"] = dict(zip(("accept_len_q", "next_token_q", "accept_len", "next_token"), results))
    return state


def run(state):
    c, seed = state["case"], state["seed"]
    if c["path"] == "lmhead":
        h, w_t, zs, tok = state["inputs"]
        out = binding.verify_fused_lmhead(h, w_t, zs, tok, c["tau_q"], MODES[c["mode_q"]], seed, 0, want_rows=c["rows"])
        return {k: v for k, v in out.items() if k != "status"}
    if c["path"] == "stage":
        zs, zl, tok = state["inputs"]
        if not (c["rows"] or c["ragged"] or c["inv_temperature"]):
            binding.verify_stage(zs, zl, tok, c["tau_q"], MODES[c["mode_q"]], seed, 0, *state["out"])
            return state["results"]
        out = binding.verify_stage_ex(zs, zl, tok, c["tau_q"], MODES[c["mode_q"]], seed, 0,
                                      n_valid=state.get("n_valid"), inv_temperature=c["inv_temperature"],
                                      want_rows=c["rows"])
        return {k: v for k, v in out.items() if k != "status"}
    zd, zq, zt, tok = state["inputs"]
    mode_q, mode_t = MODES[c["mode_q"]], MODES[c["mode_t"]]
    if c["path"] == "host":
        binding.verify_host(zd, zq, zt, tok, c["tau_q"], c["tau_t"], mode_q, seed, 0, out=state["out"])
        return state["results"]
    if mode_q == mode_t and c["div"] == "js" and not (c["rows"] or c["inv_temperature"]):
        call = binding.verify_bonus if c["bonus"] else binding.verify
        call(zd, zq, zt, tok, c["tau_q"], c["tau_t"], mode_q, seed, 0, out=state["out"])
        return state["results"]
    out = binding.verify_ex(zd, zq, zt, tok, c["tau_q"], c["tau_t"], mode_q, mode_t, seed, 0,
                            target_has_bonus_row=c["bonus"], inv_temperature=c["inv_temperature"],
                            div_kind=DIVS[c["div"]], want_rows=c["rows"], want_window=c["rows"], out=state["out"])
    rows = {k: v for k, v in out.items() if k != "status" and k not in state["out"]}
    return {"results": state["results"], **rows}


def work(case):
    B, K_d, K_q, V = case["B"], case["K_d"], case["K_q"], case["V"]
    size = 4 if case["dtype"] == "f32" else 2
    if case["path"] == "lmhead":
        M, d = B * K_d, case["d_model"]
        return {"bytes": 2 * (M * d + V * d + M * V), "flops": 2 * M * d * V}
    if case["path"] == "stage":
        n_rows = B * K_d // (2 if case["ragged"] else 1)    # half of the positions take part on average
        return {"bytes": 2 * n_rows * V * size + 4 * n_rows + 8 * B}
    # the draft's, the qualifier's and the target's rows, each once
    return {"bytes": B * (2 * K_d + K_q) * V * size + 4 * B * K_d + 16 * B}


def tolerance(case):
    # Integers: a decision within rounding of its threshold, a draw within rounding of a token boundary. Floats, against
    # 64-bit arithmetic on the same logits (divergences, residual masses, token probabilities): bf16 logits 2.4e-4
    # relative and 3.2e-4 at a single row, fp32 logits 3.9e-6 and 7.5e-6, the LM head 1.6e-6 and 2.7e-6. Four times that.
    if case["path"] == "lmhead":
        return {"rel": 7e-6, "max": 1.2e-5, "differ": 0.01}
    if case["dtype"] == "bf16":
        return {"rel": 1e-3, "max": 1.3e-3, "differ": 0.01}
    return {"rel": 1.6e-5, "max": 3e-5, "differ": 0.01}
