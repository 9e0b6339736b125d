"""What a user of the library has it do, as cases that can be timed and compared.

A case is a decoding job: a batch of prompts, a window setting, and the denoising steps that are run on it through
the binding (`State.reset`, `State.generate` or `State.step` + `State.sync`, `State.read`), from host token ids to
host token ids.  Model shapes and window settings are the ones of `synth.CONFIGS`; the other lengths are generic.

The weights are random, with one attention head of the last block and 256 rows of the LM head set by hand, so that the
model is sure of its next token, as a trained one is: it continues a sequence with (last token + 1) mod 256, and is the
surer of a masked position the closer it lies to the decoded text.  With purely random weights every confidence is
nearly the same, the ranking of the active positions hangs on the last bit, and two correct implementations decode
different texts after a few steps.

The NVFP4 option is a case of its own calls (`op_nvfp4_quantize`, `op_gemm_nvfp4` over the projections of a few blocks,
the weights quantised once): in a whole step a change of the last bit moves activations to a neighbouring 4-bit code,
and two correct implementations end a tenth apart.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2601_20332_b200 import binding as wd
from paper_2601_20332_b200 import synth


def _case(name, config, **over):
    """A case with the window setting of one of the repository's configurations, where it is not overridden."""
    c = synth.CONFIGS[config]
    case = dict(name=name, config=config, layers=c["L"], mode=c["dtype"], batch=c["batch"], prompt=c["P"], gen=c["G"],
                ragged=False, A=c["A"], B=c["B"], R=c["R"], T=c["T"], k=c["k"], steps=1, sync_each=False,
                refresh="full", stagger=False, eos=False)
    unknown = set(over) - set(case)
    if unknown:
        raise ValueError(f"unknown fields {sorted(unknown)}")
    case.update(over)
    return case


def _projections(name, config, layers, rows):
    return dict(name=name, config=config, layers=layers, mode="nvfp4", rows=rows)


def listed():
    return [
        # the smallest call: one step of the small fp32 model, as a correctness run or a demo makes it; all latency
        _case("tiny_first_step", "tiny"),
        # a whole generation of the small model, 64 tokens in 64 steps: launches and host work
        _case("tiny_generation", "tiny", steps=64),
        # time to first token: a new request with an odd prompt length, its refresh step only
        _case("llada_first_token", "llada8b", prompt=487, gen=128),
        # the headline setting: the first two phases (2 refresh + 14 normal steps) of a 256-token answer, queued
        _case("llada_generation", "llada8b", steps=16),
        # the same model late in an answer, every token handed to a reader as soon as it is there
        _case("llada_streaming", "llada8b", prompt=455, gen=57, steps=8, sync_each=True),
        # a long answer, two tokens a step, half of it decoded already
        _case("llada_long", "llada8b_long", prompt=1024, gen=512, steps=8),
        # a server's small batch of requests of different lengths whose answers end with an end-of-sequence token
        # (the window is then planned on the host, step by step)
        _case("llada_requests", "llada8b", batch=4, prompt=333, gen=256, ragged=True, steps=8, eos=True),
        # no window: every position computed and every masked one given logits, the baseline that the window replaces
        _case("llada_dense_step", "llada8b_long", A=1024, B=0, R=1, T=1),
        # eight grouped-query sequences, one phase
        _case("dream_batch", "dream7b", steps=4),
        # the same batch with its refresh steps spread over the phase, and refreshes of the window only, after an
        # odd number of decoded tokens
        _case("dream_staggered", "dream7b", prompt=701, gen=323, ragged=True, steps=8, stagger=True, refresh="window"),
        # the largest: sixteen long contexts, a wide window, a deep cut of the model
        _case("llada_wide_batch", "llada8b_sweep", layers=8, batch=16, prompt=1536, gen=1536, A=128, B=128, steps=4),
        # the 4-bit projections of a normal step (34 rows) in four blocks, more than the L2 holds
        _projections("nvfp4_projections", "llada8b", layers=4, rows=34),
    ]


_LARGEST = 0.9      # drawn cases stay below this share of the largest listed case's work


def draw(rng):
    """One more case: a model, a batch and a window from anywhere in the ranges of the listed ones."""
    def spread(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    limit = _LARGEST * max(_cost(c) for c in listed())
    while True:
        if rng.random() < 0.1:
            case = _projections("", rng.choice(["llada8b", "dream7b"]), rng.randint(3, 6), spread(1, 700))
            del case["name"]
            return case
        config = rng.choice(["tiny", "llada8b", "llada8b", "llada8b_long", "dream7b", "dream7b"])
        small = config == "tiny"
        mode = rng.choice(["f32", "bf16"]) if small else "bf16"
        batch = 1 if rng.random() < 0.5 else spread(2, 16)
        case = _case("", config, mode=mode, batch=batch, prompt=spread(17, 300 if small else 2000),
                     gen=spread(65, 200 if small else 1500), ragged=rng.random() < 0.5,
                     layers=rng.choice([2, 4, 8]) if small else spread(4, synth.CONFIGS[config]["L"]),
                     A=spread(4, 128), B=rng.randint(0, 256), R=rng.randint(1, 8), k=rng.choice([1, 1, 2]),
                     steps=rng.randint(1, 16), sync_each=rng.random() < 0.3,
                     refresh=rng.choice(["full", "full", "full", "window"]), stagger=batch > 1 and rng.random() < 0.25,
                     eos=rng.random() < 0.2)
        case["T"] = rng.randint(1, 4)
        if batch == 1 and rng.random() < 0.1:       # the baseline without a window
            case.update(A=case["gen"], B=0, R=1, refresh="full")
        del case["name"]
        if case["steps"] * case["k"] < case["gen"] and _cost(case) <= limit:
            return case


# ---------------------------------------------------------------------------------------------------------------------
# weights and inputs
# ---------------------------------------------------------------------------------------------------------------------

_ATTN_UPDATE, _FFN_UPDATE = 2.0, 0.5     # makes the two halves of a block add about a tenth of the stream's size each
_CONST, _CODE, _OUT, _BITS = 0, 1, 9, 8     # residual-stream coordinates of the copy head: a constant, a token's code, the result


def _config(case, seed):
    over = dict(L=case["layers"], wseed=seed, iseed=seed, dtype="f32" if case["mode"] == "f32" else "bf16")
    if case["config"] == "tiny" and case["mode"] == "bf16":
        over.update(dh=128, Hq=2, Hkv=2, F=704)         # the tensor-core path wants heads of 128 and widths of 64
    return synth.get_config(case["config"], **over)


def _weights(cfg):
    """synth's random weights with the usual scaling for a deep residual stream (unit embeddings, output projections
    divided by sqrt(2 L)), and the copy head written over a few of them."""
    w = synth.make_weights(cfg, device="cuda")
    L, d, dh, V = cfg["L"], cfg["d"], cfg["dh"], cfg["V"]
    half, reserved = dh // 2, _OUT + _BITS
    dev, dt = w.tok_embed.device, w.tok_embed.dtype
    code = torch.arange(V, device=dev)[:, None] >> torch.arange(_BITS, device=dev)[None, :]
    code = (2 * (code & 1) - 1).to(dt)                  # a token's low byte as eight signs
    w.tok_embed[:, :reserved] = 0.0
    w.tok_embed[:, _CONST] = 2.0
    w.tok_embed[:, _CODE:_CODE + _BITS] = 2.0 * code
    w.tok_embed[cfg["mask_id"], _CODE:_CODE + _BITS] = 0.0
    rest = w.tok_embed[:, reserved:]        # the other coordinates give every row the same norm, sqrt(d)
    fixed = w.tok_embed[:, :reserved].float().square().sum(1, keepdim=True)
    rest.mul_(((d - fixed) / rest.float().square().sum(1, keepdim=True)).sqrt().to(dt))
    for l in range(L):
        w.wo[l].mul_(_ATTN_UPDATE / math.sqrt(2 * L))
        w.w_down[l].mul_(_FFN_UPDATE / math.sqrt(2 * L))
        w.wo[l][:reserved] = 0.0
        w.w_down[l][:reserved] = 0.0
    # last block, query head 0: attends to the position before its own (with the rotary embedding, equal query and key
    # vectors rotated by one position give a score that falls off with the distance from there: about 0.6 of the weight
    # on that position, 0.2 on either neighbour), reads its code.  The faster frequencies only: the slow ones would add
    # a large constant to every score, and with it the small differences in size between the keys.
    freq = [cfg["theta"] ** (-2.0 * j / dh) for j in range(half)]
    freq = torch.tensor([f for f in freq if f > 0.02], device=dev)
    wq, wk, wv, wo = w.wq[-1], w.wk[-1], w.wv[-1], w.wo[-1]
    stream_rms = 1.0 if d < 1024 else 1.55          # of the last block's input, as measured with these weights
    strength = 0.5 * stream_rms * dh ** 0.25
    wq[:dh] = 0.0
    wk[:dh] = 0.0
    wv[:dh] = 0.0
    wq[:len(freq), _CONST] = strength
    wk[:len(freq), _CONST] = (strength * torch.cos(freq)).to(dt)
    wk[half:half + len(freq), _CONST] = (strength * torch.sin(freq)).to(dt)
    bits = torch.arange(_BITS, device=dev)
    wv[bits, _CODE + bits] = 1.0
    wo[_OUT:reserved] = 0.0
    wo[_OUT + bits, bits] = 4.0
    # LM head: token v follows a token whose low byte is v - 1
    w.lm_head[:, _OUT:reserved] = 0.0
    w.lm_head[:256] = 0.0
    w.lm_head[:256, _OUT:reserved] = code[(torch.arange(256, device=dev) - 1) % 256] * (4.0 if d < 1024 else 8.0)
    return w


def _prepare_projections(case, seed):
    cfg = _config(case, seed)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    d, F, rows = cfg["d"], cfg["F"], case["rows"]
    qkv = (cfg["Hq"] + 2 * cfg["Hkv"]) * cfg["dh"]

    def mat(n, k, scale):
        return (torch.randn(n, k, device="cuda", generator=gen) * scale).to(torch.bfloat16)

    jobs = []
    for _ in range(case["layers"]):
        for n, k in ((qkv, d), (2 * F, d), (d, F)):
            jobs.append((mat(rows, k, 1.0), wd.op_nvfp4_quantize(mat(n, k, 0.02)), n, k))
    size = max(wd.lib().wd_op_gemm_scratch_bytes(rows, n, k) for _, _, n, k in jobs)
    return dict(case=case, jobs=jobs, scratch=torch.empty(size, dtype=torch.uint8, device="cuda"))


def prepare(case, seed):
    if case["mode"] == "nvfp4":
        return _prepare_projections(case, seed)
    cfg = _config(case, seed)
    batch, S = case["batch"], case["prompt"] + case["gen"]
    ids = synth.make_prompts(cfg, batch=batch, P=case["prompt"], G=case["gen"])
    if case["ragged"]:          # requests of different lengths in one state: shorter prompts, longer answers
        for b in range(1, batch):
            ids[b, case["prompt"] - b * case["prompt"] // (3 * batch):] = cfg["mask_id"]
    rows, active = batch * S, batch * case["A"]
    ctx = wd.Context(cfg, _weights(cfg), batch, S, rows, active)
    state = wd.State(ctx, ids)
    if case["refresh"] == "window":
        state.set_refresh_mode(wd.WD_REFRESH_WINDOW)
    state.set_stagger(case["stagger"])
    if case["eos"]:
        state.set_eos(cfg["V"] - 2)         # an id that the model does not produce: the answer runs to its length
    logits = torch.zeros(active, cfg["V"], dtype=torch.float32, device="cuda")
    return dict(case=case, ctx=ctx, state=state, ids=ids, logits=logits, stream=torch.cuda.Stream())


def run(s):
    """The job: a request in, its steps, the sequences out, and of the last step also the logits of its active rows."""
    c = s["case"]
    if c["mode"] == "nvfp4":
        return [wd.op_gemm_nvfp4(wd.op_nvfp4_quantize(x), w, c["rows"], n, k, scratch=s["scratch"]) for x, w, n, k in s["jobs"]]
    st, stream = s["state"], s["stream"]
    window = c["A"], c["B"], c["R"], c["T"], c["k"]
    st.reset(s["ids"], None, stream)
    if not c["sync_each"]:
        if c["steps"] > 1:
            st.generate(*window, max_steps=c["steps"] - 1, stream=stream)
    else:
        for _ in range(c["steps"] - 1):
            st.step(*window, stream=stream)
            st.sync()
    st.set_taps(logits=s["logits"])
    _, info = st.step(*window, stream=stream)
    st.sync()
    st.set_taps()
    return dict(ids=np.stack([st.read(b)["ids"] for b in range(c["batch"])]), logits=s["logits"][:info["n_active"]])


# ---------------------------------------------------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------------------------------------------------

def _steps(case):
    """(rows, active rows, visible positions per sequence) of each step: the counts of the planner."""
    A, B, R, T, k, batch = (case[n] for n in ("A", "B", "R", "T", "k", "batch"))
    S = case["prompt"] + case["gen"]
    seqs = []
    for b in range(batch):
        cut = b * case["prompt"] // (3 * batch) if case["ragged"] else 0
        offset = b * R // batch if case["stagger"] else 0
        seqs.append(dict(decoded=case["prompt"] - cut, alive=0, vis=0, since=0, hist=[], offset=offset))
    for t in range(case["steps"]):
        rows = act = 0
        vis = []
        for q in seqs:
            refresh = t == 0 or q["since"] >= R or q["alive"] == 0 or (0 < q["offset"] < R and t == q["offset"])
            if refresh:
                q["alive"] = min(A + B, S - q["decoded"])
                q["vis"] = q["decoded"] + q["alive"]
                window_only = case["refresh"] == "window" and t > 0
                n = q["alive"] + sum(q["hist"]) if window_only else q["vis"]
                q["since"], q["hist"] = 0, []
            else:
                n = min(A, q["alive"]) + sum(q["hist"][-T:])
            a = min(A, q["alive"])
            rows, act = rows + n, act + a
            vis.append((n, q["vis"]))
            u = min(k, a)
            q["decoded"] += u
            q["alive"] -= u
            q["hist"].append(u)
            q["since"] += 1
        yield rows, act, vis


def work(case):
    """Bytes: every step reads the weights once and the keys and values of the visible positions, and writes those of
    its rows; the last step writes its logits.  Operations: the projections of the rows, the LM head of the active
    rows, the two products of the attention."""
    cfg = _config(case, 0)
    L, d, F, V = cfg["L"], cfg["d"], cfg["F"], cfg["V"]
    if case["mode"] == "nvfp4":     # 4-bit codes and a scale byte per 16 of the weights, bf16 rows in, float rows out
        rows, qkv = case["rows"], (cfg["Hq"] + 2 * cfg["Hkv"]) * cfg["dh"]
        shapes = ((qkv, d), (2 * F, d), (d, F))
        return dict(bytes=L * sum(n * k * 9 / 16 + rows * k * 2 + rows * n * 4 for n, k in shapes),
                    flops=L * sum(2 * rows * n * k for n, k in shapes))
    hq, hkv = cfg["Hq"] * cfg["dh"], cfg["Hkv"] * cfg["dh"]
    size = 4 if cfg["dtype"] == "f32" else 2
    block = d * (hq + 2 * hkv) + hq * d + 3 * d * F
    total_bytes = total_flops = act = 0
    for rows, act, vis in _steps(case):
        total_bytes += (L * block + V * d) * size + L * 2 * hkv * size * (sum(v for _, v in vis) + rows)
        total_flops += 2 * rows * L * block + 2 * act * V * d + L * sum(4 * n * v * hq for n, v in vis)
    return dict(bytes=total_bytes + act * V * 4, flops=total_flops)


def _cost(case):
    """Seconds, roughly, on a GPU of 6 TB/s and 1 PFLOP/s (fp32 at a hundredth of that), and 50 us of latency a step."""
    w = work(case)
    return (max(w["bytes"] / 6e12, w["flops"] / (1e13 if case["mode"] == "f32" else 1e15)) +
            5e-5 * case.get("steps", 1))


def tolerance(case):
    # bf16: logits of runs whose sums were taken in another order (the projections' consumers inside the GEMMs instead of
    # separate kernels) differ by 3.5e-3 to 6e-3.  fp32: 1.3e-6 from the float64 oracle.  NVFP4: equal codes on both
    # sides, float sums in another order.  Token ids are the same throughout.
    return dict(rel=0.02 if case["mode"] == "bf16" else 1e-5)
