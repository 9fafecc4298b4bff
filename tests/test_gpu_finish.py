"""The end of a step on both sides of the row count up to which a cluster of CTAs finishes a sequence (256 rows), down
to one row: wino_step leaves exactly the tokens, counts, flags and finalization steps that wino_score_rows with the
same targets followed by wino_draft_verify (its statistics read from global memory, one CTA per sequence) gives."""
import numpy as np
import pytest
import torch

import wino_synth as ws

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("draft_m", [0, 3])
@pytest.mark.parametrize("no_shadow", [False, True], ids=["verify", "no_shadow"])
@pytest.mark.parametrize("L", [1, 4, 5, 33, 63, 64, 65, 128, 129, 256, 257])
def test_step_equals_score_then_draft_verify(L, no_shadow, draft_m):
    import paper_2605_16941_gb300 as wino
    from gpu_helpers import dev
    w = ws.Workload("finish", d=64, V=3000, n_seq=3, blk_len=L, bias=((1.0, 0.0, 20.0),), predecoded=0.5, hold=0.5,
                    shadow=not no_shadow)
    W = ws.weights(w)
    st = ws.initial_state(w)
    st.tokens[1, st.blk_start:st.blk_start + L] = st.targets[1, :L]  # no MASK left in sequence 1
    Wd, H = dev(W), dev(ws.hidden_states(w, W, st))
    y = st.tokens[:, None, st.blk_start:st.blk_start + L]
    target = np.full((3, w.kinds, L), -1, np.int32)
    if not no_shadow:
        target[:, 1:] = np.where(y == w.mask_id, -1, y)
    out = []
    for whole in (True, False):
        tokens, last = dev(st.tokens), torch.zeros((3, w.seq_len), dtype=torch.int32, device="cuda")
        p = wino.make_params(w.tau1, w.tau2, w.mask_id, 3, w.seq_len, st.blk_start, L, no_shadow=no_shadow,
                             draft_m=draft_m, step_index=7, last_change=last, freeze_finished=True)
        counts = torch.full((3, 3), -5, dtype=torch.int32, device="cuda")
        flags = torch.full((3, L), -5, dtype=torch.int8, device="cuda")
        wsp = wino.workspace(w.N, w.d, w.V)
        if whole:
            wino.wino_step(H, Wd, tokens, p, counts, wsp, flags=flags)
        else:
            rows = [torch.empty(w.N, dtype=t, device="cuda") for t in (torch.int32, torch.float32, torch.float32)]
            wino.wino_score_rows(H, Wd, dev(target.reshape(-1)), *rows, wsp)
            wino.wino_draft_verify(tokens, *rows, p, counts, flags=flags)
        torch.cuda.synchronize()
        assert wino.wino_read_device_status(wsp) == wino.WINO_OK
        out.append((tokens, counts, flags, last))
    for a, b in zip(*out):
        assert torch.equal(a, b)
