"""The work whose speed is measured: passes of the ES step through the public
entry points, over the range of parameter sets, storage types, population sizes
and call patterns that programs use.

A case is a call pattern ("op") over a parameter set:

  members     the paper's loop as written: es_perturb, (rollout), es_restore
              for each member
  generation  the steady-state fused loop: one es_restore_perturb per member
              boundary, the last es_restore, then es_update_perturb, which leaves
              theta at the next generation's first member
  antithetic  pairs: perturb, flip, restore fused with the next pair's perturb,
              then es_update on the folded coefficients
  update      es_normalize_rewards, es_update_coeffs, es_update
  replay      es_replay of a seed log
  noise       es_noise_fill of one member's direction
  noalloc     es_perturb_noalloc and its restore, for programs that may not
              allocate

The caller's rollouts are left out: nothing runs between the calls.
"""
import math
import random

import numpy as np
import torch

from paper_2608_17310_gb300 import esopt as es
from paper_2608_17310_gb300 import inputs

TORCH_DTYPES = {"f32": torch.float32, "bf16": torch.bfloat16, "e4m3": torch.uint8}
NOALLOC_DTYPES = {"f32": es.ES_FP32, "bf16": es.ES_BF16}
BYTES = {"f32": 4, "bf16": 2, "e4m3": 1}


# --- the cases ---------------------------------------------------------------------

def listed():
    return [
        # the smallest set in use (65,536 fp32): a whole antithetic generation of
        # 4 pairs, where launches and the latency of one short pass count
        {"name": "quadratic_antithetic", "op": "antithetic", "layout": "single", "numel": 1 << 16,
         "dtype": "f32", "members": 4, "sigma": 0.05},
        # the same set's update over its 32 pairs: few elements, many seeds
        {"name": "quadratic_update", "op": "update", "layout": "single", "numel": 1 << 16,
         "dtype": "f32", "members": 32, "sigma": 0.05},
        # 1,048,576 fp32 parameters, 8 members, the loop as written
        {"name": "toy_members", "op": "members", "layout": "single", "numel": 1 << 20,
         "dtype": "f32", "members": 8, "sigma": 1e-3},
        # many small tensors of odd sizes (adapters, norms and biases), 8 members
        {"name": "ragged_generation", "op": "generation", "layout": "ragged", "tensors": 200,
         "largest": 150_001, "dtype": "bf16", "members": 8, "sigma": 1e-3},
        # the no-allocation entry point over one decoder layer's tensors
        {"name": "layer_noalloc", "op": "noalloc", "layout": "decoder", "layers": 1, "hidden": 2560,
         "mlp": 9728, "vocab": 0, "dtype": "bf16", "members": 1, "sigma": 1e-3},
        # one decoder layer updated by a small population
        {"name": "layer_update_n2", "op": "update", "layout": "decoder", "layers": 1,
         "hidden": 2560, "mlp": 9728, "vocab": 0, "dtype": "bf16", "members": 2, "sigma": 1e-3},
        # one member's direction regenerated for inspection, from an index that
        # starts no 16-byte block
        {"name": "noise_unaligned", "op": "noise", "layout": "single", "numel": 50_000_003,
         "start": 1_000_003, "dtype": "f32", "members": 1, "sigma": 1.0},
        # a seed log of small generations replayed over a four-layer model
        {"name": "replay_small_generations", "op": "replay", "layout": "decoder", "layers": 4,
         "hidden": 2560, "mlp": 9728, "vocab": 151_936, "dtype": "bf16", "members": 2,
         "generations": 12, "sigma": 1e-3},
        # the fused generation on a four-layer model in FP8 and its update in fp32
        {"name": "fp8_generation", "op": "generation", "layout": "decoder", "layers": 4,
         "hidden": 2560, "mlp": 9728, "vocab": 151_936, "dtype": "e4m3", "members": 4,
         "sigma": 1e-3},
        {"name": "f32_update_n16", "op": "update", "layout": "decoder", "layers": 4,
         "hidden": 2560, "mlp": 9728, "vocab": 151_936, "dtype": "f32", "members": 16,
         "sigma": 1e-3},
        # the full 4B-shaped bf16 set: a member of the loop as written, and the
        # fused generation that the benchmark times, at a small population
        {"name": "qwen4b_member", "op": "members", "layout": "decoder", "layers": 36,
         "hidden": 2560, "mlp": 9728, "vocab": 151_936, "dtype": "bf16", "members": 1,
         "sigma": 1e-3},
        {"name": "qwen4b_generation", "op": "generation", "layout": "decoder", "layers": 36,
         "hidden": 2560, "mlp": 9728, "vocab": 151_936, "dtype": "bf16", "members": 8,
         "sigma": 1e-3},
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: any call pattern, 1,000 to 10^9 parameters (odd counts
    among them), populations of 1 to 128, every storage type."""
    op = rng.choice(["members", "generation", "generation", "antithetic", "update", "update",
                     "replay", "noise", "noalloc"])
    dtype = rng.choice(["f32", "bf16", "bf16", "e4m3"])
    if op == "noise" or (op == "noalloc" and dtype == "e4m3"):
        dtype = "f32"
    layout = "single" if op == "noise" else rng.choice(["single", "ragged", "decoder"])
    c = {"op": op, "layout": layout, "dtype": dtype}
    if layout == "single":
        c["numel"] = _log_uniform(rng, 1000, 1e9)
        if op == "noise":
            c["start"] = rng.choice([0, 4 * rng.randrange(1 << 40), rng.randrange(1 << 42)])
    elif layout == "ragged":
        c["tensors"] = _log_uniform(rng, 2, 600)
        c["largest"] = _log_uniform(rng, 100, 2e6)
    else:
        c["layers"] = rng.randrange(1, 9)
        c["hidden"] = 128 * rng.randrange(1, 29)
        c["mlp"] = 2 * c["hidden"] + rng.randrange(0, 2 * c["hidden"])
        c["vocab"] = rng.choice([0, 32_003, 151_936])
    numel = _numel(c)
    c["members"] = 1 if op in ("noise", "noalloc") else max(1, min(
        _log_uniform(rng, 1, 128), int(1.2e10 / numel)))
    if op == "replay":
        c["generations"] = max(1, min(_log_uniform(rng, 2, 64),
                                      int(1.2e10 / numel / c["members"])))
    c["sigma"] = 1.0 if op == "noise" else rng.choice([5e-4, 1e-3, 0.05])
    return c


def _specs(case):
    """The parameter tensors of a case."""
    if case["layout"] == "single":
        return [inputs.TensorSpec("theta", case["numel"], "weight")]
    if case["layout"] == "ragged":
        r = random.Random(7919 * case["tensors"] + case["largest"])
        return [inputs.TensorSpec(f"t{k}", _log_uniform(r, 1, case["largest"]), "weight")
                for k in range(case["tensors"])]
    specs = inputs.qwen_shapes(case["layers"], case["hidden"], 32, 8, 128, case["mlp"],
                               max(1, case["vocab"]), tied=True)
    return specs if case["vocab"] else specs[1:]


def _numel(case):
    return sum(s.numel for s in _specs(case))


def _offsets(case):
    """Offsets of the tensors in one flat buffer, 16-byte aligned."""
    return inputs.flat_offsets(_specs(case), align=16 if case["dtype"] == "e4m3" else 8)


def _passes(case):
    """(passes over the parameters, Gaussians per parameter) of one run."""
    n = case["members"]
    return {"members": (2 * n, 2 * n),
            "generation": (n + 1, 2 * (n - 1) + 1 + n + 1),
            "antithetic": (2 * n + 2, n + 2 * (n - 1) + 2 + n),
            "update": (1, n),
            "replay": (1, n * case.get("generations", 1)),
            "noise": (0.5, 1),
            "noalloc": (2, 2)}[case["op"]]


def work(case):
    """Each call reads and writes every parameter once (es_noise_fill only
    writes; a replay needs one pass for all its generations). Per Gaussian: 9
    32-bit multiplies and about 5 additions and exclusive-ors of Philox4x32-10,
    and about 7 floating-point operations of Box-Muller and the update."""
    passes, gaussians = _passes(case)
    numel = _numel(case)
    return {"bytes": int(2 * passes * numel * BYTES[case["dtype"]]),
            "flops": int(21 * gaussians * numel)}


def tolerance(case):
    """About four times the largest difference from the 64-bit result measured
    over the listed cases and drawn ones: fp32 2.7e-7 (noise 2.3e-7), bf16
    8.2e-5 and E4M3 5e-5 at sigma 1e-3 (a few results that round to the other
    neighbour, a step of up to 2^-7 or 2^-3 of the value)."""
    if case["dtype"] == "f32":
        return {"rel": 1e-6, "max": 1e-5}
    if case["dtype"] == "bf16":
        return {"rel": 3e-4, "max": 0.02}
    return {"rel": 1e-3, "max": 0.3}


# --- inputs ------------------------------------------------------------------------

def prepare(case, seed):
    specs = _specs(case)
    rng = np.random.default_rng(seed)
    n = case["members"]
    count = n * case.get("generations", 1)
    state = {
        "case": case,
        "seeds": rng.integers(0, 1 << 63, size=count, dtype=np.uint64),
        "rewards": rng.uniform(0.0, 1.0, size=2 * n if case["op"] == "antithetic" else n),
        "sigma": case["sigma"],
        "alpha": 0.5 * case["sigma"],
    }
    if case["op"] == "noise":
        state["out"] = torch.empty(case["numel"], dtype=torch.float32, device="cuda")
        return state
    if case["dtype"] == "e4m3":
        flat, views, state["scales"] = inputs.init_params_flat_e4m3(specs, "cuda", seed=seed)
        state["flat"] = flat.view(torch.float8_e4m3fn)
    else:
        flat, views = inputs.init_params_flat(specs, TORCH_DTYPES[case["dtype"]], "cuda", seed=seed)
        state["flat"] = flat
    # every parameter's global index is its offset in the flat buffer
    bases = _offsets(case)[:-1]
    if case["op"] == "noalloc":
        state["segments"] = es.segments_from_tensors(views, bases)
        state["views"] = views
        return state
    state["plan"] = es.plan_from_tensors(views, bases, state.get("scales"))
    if case["op"] == "replay":
        state["coeffs"] = (state["alpha"] * rng.standard_normal(count) / n).astype(np.float32)
        state["counts"] = np.full(case["generations"], n, dtype=np.int32)
    return state


# --- one pass ------------------------------------------------------------------------

def run(state):
    case, seeds, sigma = state["case"], state["seeds"], state["sigma"]
    op, n = case["op"], case["members"]
    if op == "noise":
        es.es_noise_fill(int(seeds[0]), case["start"], case["numel"], state["out"])
        return state["out"]
    if op == "noalloc":
        dtype = NOALLOC_DTYPES[case["dtype"]]
        es.es_perturb_noalloc(state["segments"], dtype, int(seeds[0]), sigma)
        es.es_perturb_noalloc(state["segments"], dtype, int(seeds[0]), -sigma)
        return state["flat"]
    plan = state["plan"]
    if op == "members":
        for s in seeds:
            es.es_perturb(plan, int(s), sigma)
            es.es_restore(plan, int(s), sigma)
    elif op == "generation":
        for a, b in zip(seeds[:-1], seeds[1:]):
            es.es_restore_perturb(plan, int(a), sigma, int(b), sigma)
        es.es_restore(plan, int(seeds[-1]), sigma)
        coeffs = es.es_update_coeffs(es.es_normalize_rewards(state["rewards"]), state["alpha"],
                                     sigma)
        es.es_update_perturb(plan, seeds, coeffs, int(seeds[0]), sigma)
    elif op == "antithetic":
        es.es_perturb(plan, int(seeds[0]), sigma)
        for k in range(n):
            s = int(seeds[k])
            es.es_restore_perturb(plan, s, sigma, s, -sigma)
            if k + 1 < n:
                es.es_restore_perturb(plan, s, -sigma, int(seeds[k + 1]), sigma)
        es.es_restore(plan, int(seeds[-1]), -sigma)
        rhat = es.es_normalize_rewards(state["rewards"])
        es.es_update(plan, seeds, es.es_fold_antithetic(rhat[:n], rhat[n:], state["alpha"], sigma))
    elif op == "update":
        coeffs = es.es_update_coeffs(es.es_normalize_rewards(state["rewards"]), state["alpha"],
                                     sigma)
        es.es_update(plan, seeds, coeffs)
    else:
        es.es_replay(plan, seeds, state["coeffs"], state["counts"])
    return state["flat"]


# --- the same in 64 bits ----------------------------------------------------------------

_M32 = 0xFFFFFFFF
_CHUNK = 1 << 24


def _mul_hi_lo(m, x):
    # both factors below 2^32: the 64-bit product wraps as int64, its bits hold
    p = x * m
    return (p >> 32) & _M32, p & _M32


def _noise64(seed, start, n, device):
    """eps_seed[start .. start + n) in 64 bits: Philox4x32-10 on the block number,
    then Box-Muller on u(x) = (2 (x >> 9) + 1) / 2^24."""
    j0 = start // 4
    nb = (start + n + 3) // 4 - j0
    j = torch.arange(j0, j0 + nb, dtype=torch.int64, device=device)
    c = [j & _M32, j >> 32, torch.zeros_like(j), torch.zeros_like(j)]
    k0, k1 = seed & _M32, seed >> 32
    for _ in range(10):
        h0, l0 = _mul_hi_lo(0xD2511F53, c[0])
        h1, l1 = _mul_hi_lo(0xCD9E8D57, c[2])
        c = [h1 ^ c[1] ^ k0, l1, h0 ^ c[3] ^ k1, l0]
        k0, k1 = (k0 + 0x9E3779B9) & _M32, (k1 + 0xBB67AE85) & _M32
    u = [(2 * (x >> 9) + 1).to(torch.float64) / 16777216.0 for x in c]
    out = torch.empty(nb, 4, dtype=torch.float64, device=device)
    for q in (0, 2):
        r = torch.sqrt(-2.0 * torch.log(u[q]))
        a = 2.0 * math.pi * u[q + 1]
        out[:, q] = r * torch.cos(a)
        out[:, q + 1] = r * torch.sin(a)
    return out.reshape(-1)[start - 4 * j0:start - 4 * j0 + n]


def _store(v, dtype):
    """The nearest value of the storage type."""
    if dtype == "bf16":
        return v.to(torch.bfloat16).to(torch.float64)
    if dtype == "e4m3":
        return v.clamp(-448.0, 448.0).to(torch.float32).to(torch.float8_e4m3fn).to(torch.float64)
    return v.to(torch.float32).to(torch.float64)


def _z_score(rewards):
    r = np.asarray(rewards, dtype=np.float64)
    return (r - r.mean()) / (r.std() + 1e-8) if r.max() > r.min() else np.zeros_like(r)


def _steps(state):
    """The pass as a list of steps, each a list of (seed number, coefficient)
    that is added to theta and then rounded to the storage type."""
    case, n = state["case"], state["case"]["members"]
    s = float(np.float32(state["sigma"]))
    alpha, op = state["alpha"], case["op"]
    if op in ("members", "noalloc"):
        return [[(k, c)] for k in range(n) for c in (s, -s)]
    if op == "generation":
        steps = [[(k // 2, -s)] if k % 2 == 0 else [(k // 2 + 1, s)] for k in range(2 * n - 1)]
        coeffs = (alpha * _z_score(state["rewards"]) / n).astype(np.float32)
        return steps + [[(k, float(coeffs[k])) for k in range(n)], [(0, s)]]
    if op == "antithetic":
        steps = [[(k, c)] for k in range(n) for c in (s, -s, -s, s)]
        z = _z_score(state["rewards"])
        coeffs = (alpha * (z[:n] - z[n:]) / (2 * n)).astype(np.float32)
        return steps + [[(k, float(coeffs[k])) for k in range(n)]]
    if op == "update":
        coeffs = (alpha * _z_score(state["rewards"]) / n).astype(np.float32)
        return [[(k, float(coeffs[k])) for k in range(n)]]
    return [[(g * n + k, float(state["coeffs"][g * n + k])) for k in range(n)]
            for g in range(case["generations"])]


def exact(case, seed):
    numel = _numel(case)
    if numel * case["members"] * case.get("generations", 1) > 3.5e10:
        return None
    state = prepare(case, seed)
    seeds = [int(s) for s in state["seeds"]]
    if case["op"] == "noise":
        return torch.cat([_noise64(seeds[0], case["start"] + o, min(_CHUNK, numel - o), "cuda")
                          for o in range(0, numel, _CHUNK)])
    out = state["flat"].to(torch.float64)
    offsets, specs, steps = _offsets(case), _specs(case), _steps(state)
    owned = torch.zeros(out.numel(), dtype=torch.bool, device="cuda")  # not the padding
    scale = None if "scales" not in state else torch.ones_like(out)
    for t, spec in enumerate(specs):
        owned[offsets[t]:offsets[t] + spec.numel] = True
        if scale is not None:
            scale[offsets[t]:offsets[t] + spec.numel] = state["scales"][t]
    reused = case["op"] in ("members", "noalloc", "generation", "antithetic")
    for o in range(0, out.numel(), _CHUNK):
        v = out[o:o + _CHUNK]
        kept = [_noise64(s, o, v.numel(), "cuda") for s in seeds] if reused else None
        x = v.clone()
        for step in steps:
            total = torch.zeros_like(x)
            for k, c in step:
                total += c * (kept[k] if reused else _noise64(seeds[k], o, v.numel(), "cuda"))
            if scale is not None:
                total /= scale[o:o + _CHUNK]
            x = _store(x + total, case["dtype"])
        v.copy_(torch.where(owned[o:o + _CHUNK], x, v))
    return out
