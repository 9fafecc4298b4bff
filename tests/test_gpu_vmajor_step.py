"""wino_step on the vocabulary-major score kernel: targets from the token state, row compaction and an active-sequence
list, row-major W and the panel copy, where a tile's rows past the vocabulary lie in the next panel instead of being
filled with zeros.  The two layouts give the same bytes, and the step is the oracle's.  Sizes: one 32-column chunk and a
narrow tile; two accumulators per tile; a last round whose tiles two pairs share; several row groups.  The launch's
timeline shows that this kernel ran: its tile count is not the row-block split's."""
import numpy as np
import pytest
import torch

import oracle
import wino_synth as ws

pytestmark = pytest.mark.gpu

# (d, V, L, sequences scored with shadow rows, (groups, hw0, hw1, split) of the launch)
SHAPES = [
    (64, 47503, 15, 1, (1, 32, 0, 0)),        # 30 rows, 224-wide tiles
    (512, 59953, 24, 1, (1, 64, 0, 0)),       # 48 rows, 208-wide tiles
    (1536, 29557, 50, 3, (1, 160, 144, 0)),   # 300 rows, two accumulators
    (1536, 19999, 43, 3, (1, 144, 128, 1)),   # 258 rows, three last tiles whose accumulators go to two pairs each
    (1024, 24118, 121, 3, (3, 256, 0, 0)),    # 726 rows, three groups
]


@pytest.mark.parametrize("form", ["shadow", "compact", "active", "active_compact"])
@pytest.mark.parametrize("d,V,L,B,split", SHAPES, ids=[f"d{s[0]}_V{s[1]}_{s[3]}x{s[2]}" for s in SHAPES])
def test_step(d, V, L, B, split, form):
    import paper_2605_16941_gb300 as wino
    from gpu_helpers import compare_step, dev, host
    compact = "compact" in form
    B = B * 2 if compact else B  # one row per position: as many rows scored from twice the sequences
    n_seq = B + 2 if "active" in form else B
    # Biases up to 40 (doubled by the variant): a held token keeps its place from a logit of about ln V + 0.5 + ln 4 <= 13
    # on (p >= tau2 = 0.8 over a N(0, 1) background), so two in three of them do, also among the 7 of the smallest shape.
    w = ws.coverage_variant(ws.Workload("vmajor_step", d=d, V=V, n_seq=n_seq, blk_len=L, bias=((1.0, 0.0, 20.0),),
                                        predecoded=0.5, tau1=0.6, tau2=0.8))
    listed = list(range(n_seq))[::-1][:B] if "active" in form else list(range(n_seq))
    rows = B * L * (1 if compact else 2)
    plan = wino.wino_score_launch(rows, d, V)
    assert plan["kernel"] == 2 and (plan["n_groups"], plan["hw0"], plan["hw1"], plan["split"]) == split, plan
    assert V % plan["bn"] != 0
    by_rows = wino.wino_score_plan(rows, d, V)
    assert plan["n_groups"] * plan["n_vt"] != by_rows["n_mb"] * by_rows["n_vt"]

    W, st = ws.weights(w), ws.initial_state(w)
    H_host = ws.hidden_states(w, W, st)
    H, Wd = dev(H_host), dev(W)
    act = dev(np.array(listed, np.int32)) if "active" in form else None
    out = []
    for panels in (False, True):
        p = wino.make_params(w.tau1, w.tau2, w.mask_id, n_seq, w.seq_len, st.blk_start, L, compact=compact,
                             active_seq=act, w_panels=panels)
        tok = dev(st.tokens)
        counts = torch.full((n_seq, 3), -9, dtype=torch.int32, device="cuda")
        flags = torch.full((n_seq, L), -9, dtype=torch.int8, device="cuda")
        wsp = wino.step_workspace(p, d, V)
        Wx = wino.wino_lm_head_panels(Wd) if panels else Wd
        buf = torch.zeros(256 * wino.TIMELINE_WORDS, dtype=torch.int64, device="cuda")
        torch.cuda.synchronize()
        wino.wino_timeline_begin(buf, 1, 256)
        try:
            wino.wino_step(H, Wx, tok, p, counts, wsp, flags=flags)
            torch.cuda.synchronize()
        finally:
            wino.wino_timeline_end()
        assert wino.wino_read_device_status(wsp) == wino.WINO_OK
        T = buf.view(256, wino.TIMELINE_WORDS).cpu().numpy().view(np.uint64)
        assert int((T[0::2, 7] & np.uint64(0xFFFFFFFF)).sum()) == plan["n_groups"] * plan["n_vt"]
        out.append((tok, counts, flags, wsp))
    for a, b, what in zip(*out, ("tokens", "counts", "flags", "workspace")):
        assert torch.equal(a, b), f"{what} differ between row-major W and its panel copy"

    tok, cnt, fl = (host(x) for x in out[0][:3])
    others = [s for s in range(n_seq) if s not in listed]
    assert np.array_equal(tok[others], st.tokens[others]) and np.all(cnt[others] == -9) and np.all(fl[others] == -9)
    per_seq = 2 * L
    H_sub = np.concatenate([H_host[s * per_seq:(s + 1) * per_seq] for s in listed])
    o = oracle.step(H_sub, W, st.tokens[listed], st.blk_start, L, w.mask_id, w.tau1, w.tau2)
    rep = compare_step(st.tokens[listed], tok[listed], cnt[listed], o, st.blk_start, L, w.mask_id, w.tau1, w.tau2)
    assert rep["drafted"] > 0 and rep["kept_decoded"] > 0 and rep["remasked"] > 0, rep
