"""Timed cases of this framework: denoising steps and decodes of the masked-diffusion model, with and without the
key/value caches, and the training of the filter.  Each case goes through the public entry points (`binding.Decoder`,
the C ABI's `l2pd_denoise_step`, `binding.filter_train*`).

Models: the tiny fp32 model and the LLaDA-8B shape of `workloads`, and a small bf16 model with heads of 64, the one
head size that runs another attention kernel.

The bf16 models are random-init, so the two best logits of a row often lie closer together than bf16 resolves, and a
decode would follow a rounding.  What is decided is therefore made independent of near-ties, without changing the work:
  * the LM head's bias lifts one frequent token, drawn from the seed (its confidence then spreads around 0.8),
    so that the argmax does not hang on a rounding; the step cases also return all logits;
  * the filter is a two-layer MLP of the usual shape that passes the next group of positions once the group before
    it is committed (committed positions read 1.0): eight steps a block, a usual number.
The fp32 model keeps its natural logits and the noisy-identity filter of `workloads`.
"""
import ctypes
import math

import numpy as np
import torch

from paper_2509_25188_b200 import binding, workloads as wl

DEVICE = "cuda:0"
TAU = 0.96
SMALL = wl.ModelShape(n_layers=4, d_model=512, n_heads=8, head_dim=64, d_ff=1376, vocab=8192, rms_eps=1e-5,
                      rope_theta=10000.0, mask_id=8191, eot_id=8190, dtype="bf16")
SHAPES = {"tiny": wl.TINY, "small": SMALL, "llada8b": wl.LLADA_8B}
GROUPS = 8                 # groups of positions a block is committed in, hence steps of a block
NO_CACHE, PREFIX, DUAL = 0, 1, 2


def _decode(name, model, batch, prompt, gen, block, cache=NO_CACHE):
    return {"name": name, "kind": "decode", "model": model, "batch": batch, "prompt": prompt, "gen": gen, "block": block,
            "cache": cache}


def _block(name, batch, prompt, gen, block, cache, steps):
    return {"name": name, "kind": "block", "model": "llada8b", "batch": batch, "prompt": prompt, "gen": gen,
            "block": block, "cache": cache, "steps": steps}


def _train(name, samples, s, layers, batch, epochs):
    return {"name": name, "kind": "train", "samples": samples, "s": s, "layers": layers, "batch": batch, "epochs": epochs}


def listed():
    return [
        # the smallest model and call: a whole fp32 decode, bound by launches and latency
        _decode("decode fp32 tiny 1x(32+64)", "tiny", 1, 32, 64, 16),
        # a small bf16 model with heads of 64, two ragged sequences
        _decode("decode bf16 small 2x(57+96)", "small", 2, 57, 96, 32),
        # a short question and answer on the 8B shape: fewer rows than one 128-row tile, no cache
        _decode("decode 8b short 1x(61+64)", "llada8b", 1, 61, 64, 32),
        # the usual single request: 256 + 256, one whole-sequence step
        _block("step 8b 1x(256+256)", 1, 256, 256, 32, NO_CACHE, 1),
        # the same request as a whole decode with the dual cache: 64 steps, 56 of them over 32 rows
        _decode("decode 8b dual 1x(256+256)", "llada8b", 1, 256, 256, 32, DUAL),
        # a few requests of odd length together
        _block("step 8b 3x(183+160)", 3, 183, 160, 32, NO_CACHE, 1),
        # a server's batch, no cache
        _block("step 8b 16x(512+512)", 16, 512, 512, 32, NO_CACHE, 1),
        # long prompts and answers with the prefix cache: a block's first step and two cached ones
        _block("block 8b prefix 8x(1024+1024)", 8, 1024, 1024, 32, PREFIX, 3),
        # the same with the dual cache: a whole block
        _block("block 8b dual 8x(1024+1024)", 8, 1024, 1024, 32, DUAL, GROUPS),
        # filter training at the size the method is trained at: 2,640 prompts x 32 steps, full batch
        _train("train filter 84480x32", 84480, 32, 2, 0, 200),
        # a deeper filter for blocks of 64, in mini-batches
        _train("train filter 6000x64 deep", 6000, 64, 4, 1024, 10),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["decode", "decode", "step", "step", "step", "block", "block", "train"])
    if kind == "decode":
        model = rng.choice(["tiny", "small", "llada8b", "llada8b"])
        block = 16 if model == "tiny" else rng.choice([16, 32, 32, 64])
        batch = rng.randint(1, 3)
        if model == "llada8b":
            # at most 16 steps over some hundred rows without a cache, 64 with the dual one
            cache = rng.choice([NO_CACHE, DUAL])
            gen = block * (rng.randint(2, 6) if cache else 2)
            prompt = _log_int(rng, 24, 256)
        else:
            cache, gen, prompt = rng.choice([NO_CACHE, PREFIX, DUAL]), block * rng.randint(2, 4), _log_int(rng, 9, 96)
        case = _decode("", model, batch, prompt, gen, block, cache)
    elif kind in ("step", "block"):
        block = rng.choice([16, 32, 32, 64])
        rows = _log_int(rng, 160, 14000)
        batch = min(16 if kind == "step" else 8, max(1, int(rows / _log_int(rng, 160, 2000))))
        seq = max(2 * block + 8, min(2048, rows // batch))
        gen = block * max(1, int(seq * rng.uniform(0.2, 0.7)) // block)
        prompt = seq - gen
        if kind == "step":
            case = _block("", batch, prompt, gen, block, NO_CACHE, 1)
        else:
            cache = rng.choice([PREFIX, DUAL])
            case = _block("", batch, prompt, gen, block, cache, 3 if cache == PREFIX else rng.randint(3, GROUPS))
    else:
        s, layers = rng.choice([(32, 2), (32, 2), (16, 2), (27, 2), (32, 4), (64, 2), (48, 1)])
        samples = _log_int(rng, 2000, 80000)
        batch = rng.choice([0, 0, 0, 1024, 4096])
        updates_per_epoch = -(-samples // batch) if batch else 1
        case = _train("", samples, s, layers, batch, max(1, 60 // updates_per_epoch))
    del case["name"]
    return case


# ---- inputs ------------------------------------------------------------------------------------------------------

def _weights(shape, seed):
    """N(0, 0.02^2) matrices drawn on the device in the model's type; norm gains 1 (fp32: the final gain that spreads
    the logits)."""
    g = torch.Generator(device=DEVICE)
    g.manual_seed(seed)
    dtype = torch.bfloat16 if shape.dtype == "bf16" else torch.float32
    d, f, v, hd = shape.d_model, shape.d_ff, shape.vocab, shape.n_heads * shape.head_dim

    def mat(rows, cols):
        return torch.randn(rows, cols, generator=g, device=DEVICE, dtype=dtype).mul_(0.02)

    ones = torch.ones(d, device=DEVICE)
    layers = [{"wqkv": mat(3 * hd, d), "wo": mat(d, hd), "w_gate": mat(f, d), "w_up": mat(f, d), "w_down": mat(d, f),
               "norm1": ones, "norm2": ones} for _ in range(shape.n_layers)]
    gain = wl.spread_gain(shape) if shape.dtype == "fp32" else 1.0
    return {"tok_emb": mat(v, d), "lm_head": mat(v, d), "final_norm": torch.full((d,), gain, device=DEVICE),
            "layers": layers}


def _token_bias(shape, rng):
    """A token prior as wide as the logits themselves, and one frequent token lifted above the rest's log-sum-exp."""
    sigma = 0.02 * math.sqrt(shape.d_model)       # deviation of a logit of a unit-RMS row
    bias = (rng.standard_normal(shape.vocab) * sigma).astype(np.float32)
    bias[rng.integers(0, min(shape.mask_id, shape.eot_id))] = math.log(shape.vocab) + sigma ** 2 + 1.5
    return bias


def _group_filter(s, rng):
    """relu(1000 c - 999) is 1 for a committed position and 0 below 0.999; a group passes (logit 8 above tau's) once
    the last position of the group before it reads 1, the first group always."""
    size = max(1, s // GROUPS)
    base = math.log(TAU / (1.0 - TAU))
    w1 = (1000.0 * np.eye(s)).astype(np.float32)
    w2 = (rng.standard_normal((s, s)) * 0.02).astype(np.float32)
    b2 = np.full(s, base - 8.0, np.float32)
    for j in range(s):
        first = (j // size) * size
        if first == 0:
            b2[j] = base + 8.0
        else:
            w2[j, first - 1] += 16.0
    return {"w1": w1, "b1": np.full(s, -999.0, np.float32), "w2": w2, "b2": b2}


def _prepare_train(case, seed):
    rng = np.random.default_rng(seed)
    s, layers = case["s"], case["layers"]
    c = torch.rand(case["samples"], s, generator=torch.Generator(device=DEVICE).manual_seed(seed), device=DEVICE)
    noise = torch.randn(case["samples"], s, generator=torch.Generator(device=DEVICE).manual_seed(seed + 1), device=DEVICE)
    y = (c + 0.15 * noise > 0.6).to(torch.uint8)
    eye = np.eye(s)
    params = [((eye + rng.standard_normal((s, s)) * 0.5 / math.sqrt(s)).astype(np.float32),
               (rng.standard_normal(s) * 0.02).astype(np.float32)) for _ in range(layers)]
    return {"case": case, "c": c, "y": y, "layers": params}


def prepare(case, seed):
    if case["kind"] == "train":
        return _prepare_train(case, seed)
    shape, B, P, G, s = SHAPES[case["model"]], case["batch"], case["prompt"], case["gen"], case["block"]
    rng = np.random.default_rng(seed)
    fp32 = shape.dtype == "fp32"
    filt = wl.make_filter(s, TAU, seed=seed) if fp32 else _group_filter(s, rng)
    dec = binding.Decoder(shape, _weights(shape, seed), filt, block_len=s, tau=TAU, kv_cache=case["cache"], max_batch=B,
                          max_seq=P + G, committed_conf_mode=0 if fp32 else 1,
                          lm_head_bias=None if fp32 else _token_bias(shape, rng))
    prompts = rng.integers(0, min(shape.mask_id, shape.eot_id), size=(B, P)).astype(np.int32)
    state = {"case": case, "dec": dec, "prompts": prompts}
    if case["kind"] == "block":
        state["d_prompts"] = torch.from_numpy(prompts).to(DEVICE)
        state["outs"] = [{"conf": torch.zeros(B, s, device=DEVICE),
                          "pred": torch.zeros(B, s, dtype=torch.int32, device=DEVICE),
                          "p": torch.zeros(B, s, device=DEVICE),
                          "unmask": torch.zeros(B, s, dtype=torch.uint8, device=DEVICE)} for _ in range(case["steps"])]
        state["outs"][-1]["logits"] = torch.zeros(B, s, shape.vocab, device=DEVICE)
    return state


# ---- one pass ----------------------------------------------------------------------------------------------------

def _denoise_step(dec, out):
    """l2pd_denoise_step of the C ABI into the caller's device buffers."""
    logits = out.get("logits")
    o = binding.StepOut(d_conf=out["conf"].data_ptr(), d_pred=out["pred"].data_ptr(), d_p=out["p"].data_ptr(),
                        d_unmask=out["unmask"].data_ptr(), d_logits=logits.data_ptr() if logits is not None else None)
    status = binding.lib.l2pd_denoise_step(dec.ctx, torch.cuda.current_stream().cuda_stream, ctypes.byref(o))
    if status:
        raise binding.L2pdError(status, binding.lib.l2pd_last_error(dec.ctx).decode())


def run(state):
    case = state["case"]
    if case["kind"] == "decode":
        tokens, out_len, steps, total = state["dec"].decode(state["prompts"], case["gen"])
        return {"tokens": tokens, "out_len": out_len, "steps": steps, "total_steps": total}
    if case["kind"] == "block":
        dec = state["dec"]
        dec.state_reset_device(state["d_prompts"], case["gen"])
        for out in state["outs"]:
            _denoise_step(dec, out)
        return state["outs"]
    if case["layers"] == 2:
        (w1, b1), (w2, b2) = state["layers"]
        return binding.filter_train({"w1": w1, "b1": b1, "w2": w2, "b2": b2}, state["c"], state["y"], case["epochs"],
                                    batch_size=case["batch"])
    return binding.filter_train_layers(state["layers"], state["c"], state["y"], case["epochs"], batch_size=case["batch"])


# ---- what a pass cannot do without -------------------------------------------------------------------------------

def _step_work(shape, batch, rows, keys, block, cached, writes_store):
    """One step over `rows` rows of each sequence against `keys` keys: every weight and stored key / value read once."""
    d, f, v, nl, hd = shape.d_model, shape.d_ff, shape.vocab, shape.n_layers, shape.n_heads * shape.head_dim
    size = 2 if shape.dtype == "bf16" else 4
    params = nl * (4 * d * hd + 3 * d * f) + v * d
    flops = 2.0 * batch * rows * nl * (4 * d * hd + 3 * d * f) + 4.0 * nl * hd * batch * rows * keys + 2.0 * batch * block * d * v
    store = 2.0 * size * nl * hd * batch
    return {"bytes": size * params + size * batch * rows * d + (store * keys if cached else store * rows if writes_store else 0.0),
            "flops": flops}


def work(case):
    if case["kind"] == "train":
        s, n, epochs, layers = case["s"], case["samples"], case["epochs"], case["layers"]
        # per sample and layer: one product forward, one for the weights' gradient, and one for the layer below's
        return {"bytes": epochs * 5.0 * n * s, "flops": 2.0 * s * s * n * epochs * (3 * layers - 1)}
    shape, B, P, G, s, cache = SHAPES[case["model"]], case["batch"], case["prompt"], case["gen"], case["block"], case["cache"]
    L = P + G
    if case["kind"] == "block":
        blocks, per_block = 1, case["steps"]
    else:
        blocks, per_block = G // s, GROUPS
    total = {"bytes": 0.0, "flops": 0.0}
    for b in range(blocks):
        for i in range(per_block):
            in_block = cache != NO_CACHE and i > 0
            rows = L if not in_block else (L - P - b * s if cache == PREFIX else s)
            w = _step_work(shape, B, rows, L, s, in_block, cache != NO_CACHE)
            total = {k: total[k] + w[k] for k in total}
    if case["kind"] == "block":
        total["bytes"] += 4.0 * B * s * shape.vocab            # the logits come out once
    return total


def tolerance(case):
    """Measured: the path against itself with its sums in another order (K slices added in completion order, the rotation
    as a kernel of its own, the other attention kernel), and the training against itself in 64 bits."""
    if case["kind"] == "train":
        # 64 bits: up to 9e-5 and 6e-4 (a gradient near zero decides the sign of an early update), mostly 2e-6
        return {"rel": 4e-4, "max": 1e-2}
    if case["model"] == "tiny":
        return {"rel": 1e-5, "differ": 1e-3}
    # 32 layers of random weights amplify a rounding: logits up to 1.4e-2 apart (largest difference 0.07), confidences
    # 8e-3; 3e-2 rather than four times that, since ids and decisions have to agree as well
    return {"rel": 3e-2, "max": 0.4, "differ": 1e-3}
