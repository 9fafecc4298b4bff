"""Measured cases: what users of the WINO step library run, through its public entry points.

Four kinds of call, each with the inputs a decoding program has in hand:

  step    one wino_step: the current block's rows and its shadow rows through the LM head, the vocabulary
          softmax and the in-place draft / verify / re-mask update (plus its options: WINO+ block rows only,
          row compaction, a list of active sequences, fixed-M drafting).  Returns the token state, counts, flags.
  score   wino_score_rows on the row-major LM head: argmax, largest probability, target probability and, on
          request, the entropy of every row (evaluation, distillation targets, other decoding rules).
  decode  wino_decode: the block loop run by the library, one host read of the counts per step.
  panels  wino_lm_head_panels: the LM head's panel copy, made when a head is loaded or changed.

Hidden states are N(0, 1) noise plus a planted token whose logit is raised by a bias drawn per row; the LM head is
N(0, 1/d); everything bf16.  Half of the pre-decoded positions hold their planted token, so drafting by threshold,
the at-least-one rule, kept and re-masked positions all occur.
"""
import math

import torch

import paper_2605_16941_gb300 as wino

HEAD = {"d": 4096, "V": 126464}  # the repository's LLaDA-shaped head
PROMPT = 32


def listed():
    step = {"kind": "step", **HEAD, "panels": True}
    return [
        # The smallest call: a toy head, where launches and latency are all there is.
        {"name": "step_tiny", "kind": "step", "d": 64, "V": 1000, "panels": True, "n_seq": 1, "blk_len": 32},
        # One interactive session: a 32-token block of one sequence, 64 rows; the LM head's bytes are the cost.
        {**step, "name": "step_b1_l32", "n_seq": 1, "blk_len": 32},
        # One sequence with a long block (the repository's single-sequence benchmark), 256 rows.
        {**step, "name": "step_b1_l128", "n_seq": 1, "blk_len": 128},
        # A few sessions batched, sizes that fit no tile: 3 sequences of 50 positions, 300 rows.
        {**step, "name": "step_b3_l50", "n_seq": 3, "blk_len": 50},
        # The batched decode step of the repository's loop configuration: 1024 rows.
        {**step, "name": "step_b16_l32", "n_seq": 16, "blk_len": 32},
        # The largest: the unified text + image vocabulary, 4 sequences of 256 positions, 2048 rows.
        {"name": "step_unified_b4_l256", "kind": "step", "d": 4096, "V": 134400, "panels": True, "n_seq": 4,
         "blk_len": 256},
        # WINO+ inference: no shadow rows, 128 block rows.
        {**step, "name": "step_plus_b1_l128", "n_seq": 1, "blk_len": 128, "no_shadow": True},
        # A server late in a block: 11 of 16 sequences still decode, one row per position: 352 rows.
        {**step, "name": "step_active_b16_l32", "n_seq": 16, "blk_len": 32, "n_active": 11, "compact": True},
        # Evaluation of hidden states on a row-major head of odd size, with entropy.
        {"name": "score_entropy_n1000", "kind": "score", "d": 1536, "V": 100003, "N": 1000, "entropy": True},
        # A small model's head, row-major, an ordinary ragged batch.
        {"name": "score_small_n333", "kind": "score", "d": 1024, "V": 32000, "N": 333, "entropy": False},
        # A whole decode of 2 blocks of 32 positions in 4 sequences, the counts read back after every step.
        {"name": "decode_b4_l32", "kind": "decode", **HEAD, "panels": True, "n_seq": 4, "blk_len": 32, "n_blocks": 2,
         "waves": 4},
        # A new LM head is loaded and its panel copy made.
        {"name": "panels_llada", "kind": "panels", **HEAD},
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _blocks(rng, rows):
    """n_seq sequences of blk_len positions, n_seq * blk_len <= rows."""
    blk_len = _log_int(rng, 4, min(256, rows))
    return _log_int(rng, 1, max(1, rows // blk_len)), blk_len


def draw(rng):
    kind = rng.choices(["step", "score", "decode", "panels"], [10, 6, 2, 1])[0]
    d, V = 64 * _log_int(rng, 1, 64), _log_int(rng, 1000, 134400)
    if kind == "panels":
        return {"kind": kind, "d": d, "V": V}
    if rng.random() < 0.4:  # the large heads are the ordinary ones
        d, V = 4096, rng.choice([126464, 134400])
    if kind == "score":
        if rng.random() < 0.3:
            d -= 8 * rng.randint(1, 7)  # any multiple of 8
        return {"kind": kind, "d": d, "V": V, "N": _log_int(rng, 1, 2048), "entropy": rng.random() < 0.5}
    if kind == "decode":
        n_seq, blk_len = _blocks(rng, 128)
        return {"kind": kind, "d": d, "V": V, "panels": True, "n_seq": n_seq, "blk_len": blk_len,
                "n_blocks": rng.randint(1, 2), "waves": rng.randint(1, 4)}
    n_seq, blk_len = _blocks(rng, 1024)
    case = {"kind": kind, "d": d, "V": V, "panels": rng.random() < 0.8, "n_seq": n_seq, "blk_len": blk_len}
    option = rng.choice(["", "", "no_shadow", "compact", "active", "active_compact", "fixed_m"])
    if option == "no_shadow":
        case["no_shadow"] = True
    if option == "fixed_m":
        case["draft_m"] = _log_int(rng, 1, blk_len)
    if option.endswith("compact"):
        case["compact"] = True
    if option.startswith("active"):
        case["n_active"] = rng.randint(1, n_seq)
    return case


# ---------------------------------------------------------------- inputs

def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(seed)


def _head(case, g):
    """W [V, d] ~ N(0, 1/d), bf16."""
    return torch.randn((case["V"], case["d"]), generator=g, device="cuda", dtype=torch.bfloat16) / math.sqrt(case["d"])


def _hidden(W, planted, bias, g):
    """[rows, d] bf16: unit noise, with the planted token's logit of each row raised by about `bias`."""
    h = torch.randn((planted.numel(), W.shape[1]), generator=g, device="cuda", dtype=torch.float32)
    w = W[planted].float()
    return (h + (bias / w.square().sum(1)).unsqueeze(1) * w).to(torch.bfloat16)


def _ints(lo, hi, shape, g):
    return torch.randint(lo, hi, shape, generator=g, device="cuda", dtype=torch.int64)


def _uniform(lo, hi, n, g):
    return lo + (hi - lo) * torch.rand(n, generator=g, device="cuda")


def prepare(case, seed):
    return {"step": _prepare_step, "score": _prepare_score, "decode": _prepare_decode,
            "panels": _prepare_panels}[case["kind"]](case, seed)


def _lm_head(W, panels):
    return wino.wino_lm_head_panels(W) if panels else W


def _prepare_step(case, seed):
    g = _generator(seed)
    B, L, V, mask = case["n_seq"], case["blk_len"], case["V"], case["V"] - 1
    kinds = 1 if case.get("no_shadow") else 2
    W = _head(case, g)
    target = _ints(0, mask, (B, L), g)
    H = _hidden(W, target[:, None, :].expand(B, kinds, L).reshape(-1), _uniform(0.0, 20.0, B * kinds * L, g), g)
    tokens = torch.full((B, PROMPT + 2 * L), mask, dtype=torch.int32, device="cuda")
    tokens[:, :PROMPT] = _ints(0, mask, (B, PROMPT), g).int()
    u = torch.rand((B, L), generator=g, device="cuda")  # 20 % hold their planted token, 20 % a random one, 60 % MASK
    other = _ints(0, mask, (B, L), g)
    tokens[:, PROMPT:PROMPT + L] = torch.where(u < 0.2, target, torch.where(u < 0.4, other, mask)).int()
    active = None
    if case.get("n_active"):
        active = torch.randperm(B, generator=g, device="cuda")[:case["n_active"]].sort().values.int()
    params = wino.make_params(0.7, 0.9, mask, B, PROMPT + 2 * L, PROMPT, L, no_shadow=bool(case.get("no_shadow")),
                              compact=bool(case.get("compact")), draft_m=case.get("draft_m", 0), active_seq=active,
                              w_panels=case["panels"])
    return {"case": case, "H": H, "W": _lm_head(W, case["panels"]), "tokens": tokens, "params": params,
            "active": active, "counts": torch.zeros((B, 3), dtype=torch.int32, device="cuda"),
            "flags": torch.zeros((B, L), dtype=torch.int8, device="cuda"),
            "ws": wino.step_workspace(params, case["d"], V)}


def _score_inputs(case, seed):
    g = _generator(seed)
    N, V = case["N"], case["V"]
    W = _head(case, g)
    planted = _ints(0, V, (N,), g)
    H = _hidden(W, planted, _uniform(0.0, 20.0, N, g), g)
    # the probability of the planted token (the likely one), of a random token, or of none
    u = torch.rand(N, generator=g, device="cuda")
    target = torch.where(u < 0.6, planted, torch.where(u < 0.9, _ints(0, V, (N,), g), -1)).int()
    return H, W, target


def _prepare_score(case, seed):
    H, W, target = _score_inputs(case, seed)
    out = lambda dtype: torch.empty(case["N"], dtype=dtype, device="cuda")  # noqa: E731
    return {"case": case, "H": H, "W": W, "target": target, "argmax": out(torch.int32), "pmax": out(torch.float32),
            "ptarget": out(torch.float32), "entropy": out(torch.float32) if case["entropy"] else None,
            "ws": wino.workspace(case["N"], case["d"], case["V"])}


def _ready_at(case):
    """Per position: the step of its block from which it is confident, and whether it is first drafted wrongly."""
    L = case["blk_len"]
    return [l % min(case["waves"], L) for l in range(L)], [l % 7 == 3 for l in range(L)]


def _block_steps(case):
    """Steps until a block has no MASK: a wrongly drafted position is re-masked and drafted again."""
    at, wrong = _ready_at(case)
    return max(a + (3 if w else 1) for a, w in zip(at, wrong))


def _prepare_decode(case, seed):
    g = _generator(seed)
    B, L, V, nb, mask = case["n_seq"], case["blk_len"], case["V"], case["n_blocks"], case["V"] - 1
    W = _head(case, g)
    at, wrong = (torch.tensor(x, device="cuda") for x in _ready_at(case))
    hidden = []
    for _ in range(nb):
        # a wrong token first, then the right one: the two differ
        first = _ints(0, mask, (B, L), g)
        right = (first + _ints(1, mask, (B, L), g)) % mask
        for k in range(_block_steps(case)):
            planted = torch.where(wrong & (at >= k), first, right)
            bias = torch.where(at <= k, 30.0, 0.0).expand(B, L)
            both = lambda x: x[:, None, :].expand(B, 2, L).reshape(-1)  # noqa: E731  block rows, shadow rows
            hidden.append(_hidden(W, both(planted), both(bias), g))
    S = PROMPT + nb * L
    tokens = torch.full((B, S), mask, dtype=torch.int32, device="cuda")
    tokens[:, :PROMPT] = _ints(0, mask, (B, PROMPT), g).int()
    last_change = torch.zeros((B, S), dtype=torch.int32, device="cuda")
    params = wino.make_params(0.7, 0.9, mask, B, S, PROMPT, L, max_steps=_block_steps(case) + 8, freeze_finished=True,
                              last_change=last_change, w_panels=case["panels"])
    return {"case": case, "hidden": hidden, "W": _lm_head(W, case["panels"]), "prompt": tokens, "params": params,
            "last_change": last_change, "counts": torch.zeros((B, 3), dtype=torch.int32, device="cuda"),
            "counts_host": torch.zeros((B, 3), dtype=torch.int32, pin_memory=True),
            "ws": wino.step_workspace(params, case["d"], V)}


def _prepare_panels(case, seed):
    W = _head(case, _generator(seed))
    return {"case": case, "W": W, "Wp": torch.empty((case["d"] // 64, case["V"], 64), dtype=W.dtype, device="cuda")}


# ---------------------------------------------------------------- one pass

def run(s):
    kind = s["case"]["kind"]
    if kind == "step":
        wino.wino_step(s["H"], s["W"], s["tokens"], s["params"], s["counts"], s["ws"], flags=s["flags"])
        return {"tokens": s["tokens"], "counts": s["counts"], "flags": s["flags"]}
    if kind == "score":
        wino.wino_score_rows(s["H"], s["W"], s["target"], s["argmax"], s["pmax"], s["ptarget"], s["ws"],
                             entropy=s["entropy"])
        return {"argmax": s["argmax"], "pmax": s["pmax"], "ptarget": s["ptarget"], "entropy": s["entropy"]}
    if kind == "decode":
        tokens = s["prompt"].clone()  # a new request
        s["last_change"].zero_()
        status, blocks, _ = wino.wino_decode(s["W"], tokens, s["params"], s["case"]["n_blocks"],
                                             lambda k, blk_start: s["hidden"][min(k, len(s["hidden"]) - 1)],
                                             s["counts"], s["counts_host"], s["ws"])
        return {"tokens": tokens, "last_change": s["last_change"], "blocks": [list(b) for b in blocks],
                "status": int(status)}
    return wino.wino_lm_head_panels(s["W"], s["Wp"])


# ---------------------------------------------------------------- what a pass cannot do without

def work(case):
    d, V = case["d"], case["V"]
    if case["kind"] == "panels":
        return {"bytes": 4 * d * V, "flops": 0}
    if case["kind"] == "score":
        N = case["N"]
        return {"bytes": 2 * d * (V + N) + 4 * N * (5 if case["entropy"] else 4), "flops": 2 * N * d * V}
    n_seq, L = case.get("n_active") or case["n_seq"], case["blk_len"]
    rows = n_seq * L * (1 if case.get("no_shadow") or case.get("compact") else 2)
    # tokens of the block read and written, flags and counts written
    step = {"bytes": 2 * d * (V + rows) + n_seq * (9 * L + 12), "flops": 2 * rows * d * V}
    n = case["n_blocks"] * _block_steps(case) if case["kind"] == "decode" else 1
    return {k: n * v for k, v in step.items()}


def tolerance(case):
    if case["kind"] == "panels":
        return "exact"
    if case["kind"] == "score":
        # fp32 logits of up to 4096 products, fp32 exponentials and sums
        return {"rel": 2e-5, "max": 2e-4, "differ": 0.005}
    # Whole numbers; a decision within rounding of a threshold, or a near-tie of two logits, may go either way.
    return {"rel": 0.0, "differ": 0.005}


def exact(case, seed):
    if case["kind"] != "score":
        return None  # the other kinds return whole numbers and copies
    H, W, target = _score_inputs(case, seed)
    N, V = case["N"], case["V"]
    h = H.double()
    logits = torch.empty((N, V), dtype=torch.float64, device="cuda")
    for v in range(0, V, 16384):
        logits[:, v:v + 16384] = h @ W[v:v + 16384].double().T
    top, argmax = logits.max(1)
    at = logits.gather(1, target.clamp(min=0).long().unsqueeze(1)).squeeze(1)
    logits -= top.unsqueeze(1)
    e = logits.exp()
    z = e.sum(1)
    ptarget = torch.where(target >= 0, (at - top).exp() / z, 0.0)
    entropy = z.log() - (e * logits).sum(1) / z if case["entropy"] else None
    return {"argmax": argmax.int(), "pmax": 1.0 / z, "ptarget": ptarget, "entropy": entropy}
