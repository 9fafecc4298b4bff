"""A step writes nothing outside the workspace that wino_workspace_size_step asks for, however few of the batch's
sequences it scores: a workspace of exactly that size inside a guarded buffer, with far more sequences in the batch than
the workspace has tickets for.  The listed sequences come out as in a step over a batch of just those, the others stay
as they were."""
import numpy as np
import pytest
import torch

import wino_synth as ws

pytestmark = pytest.mark.gpu

GUARD = 1 << 16  # bytes on either side; more than 4 bytes per sequence of every batch below


# (n_seq, listed sequences, blk_len, options)
CASES = [
    (4096, [17], 4, {"compact": True}),            # 4 scored rows: 64 tickets reserved
    (512, [511], 4, {"compact": True}),            # the gathered rows lie within 4 * n_seq bytes of the tickets
    (4096, [4095, 0, 77], 1, {}),
    (700, [699, 3], 129, {}),                      # 258 rows per sequence: tickets are used, 2 of 320 reserved
    (4096, [5, 4000], 1, {"no_shadow": True}),
    (4096, None, 1, {"no_shadow": True}),          # every sequence, one row each: 2048 tickets reserved
]


@pytest.mark.parametrize("n_seq,listed,L,opts", CASES, ids=[f"s{c[0]}_a{len(c[1] or [])}_L{c[2]}" + "".join(
    "_" + o for o in c[3]) for c in CASES])
def test_step_stays_inside_its_workspace(n_seq, listed, L, opts):
    import paper_2605_16941_gb300 as wino
    from gpu_helpers import dev
    w = ws.Workload("bounds", d=64, V=1000, n_seq=n_seq, blk_len=L, bias=((1.0, 0.0, 16.0),), predecoded=0.5, hold=0.5,
                    prompt_len=3, shadow=not opts.get("no_shadow", False))
    W = ws.weights(w)
    st = ws.initial_state(w)
    Wd, H, tokens0 = dev(W), dev(ws.hidden_states(w, W, st)), dev(st.tokens)
    act = None if listed is None else dev(np.array(listed, np.int32))

    def params(n, **kw):
        return wino.make_params(w.tau1, w.tau2, w.mask_id, n, w.seq_len, st.blk_start, L, **opts, **kw)

    def outputs(n):
        return (torch.full((n, 3), -9, dtype=torch.int32, device="cuda"),
                torch.full((n, L), -9, dtype=torch.int8, device="cuda"))

    p = params(n_seq, active_seq=act)
    size = wino.wino_workspace_size_step(p, w.d, w.V)
    assert size % 256 == 0
    buf = torch.full((GUARD + size + GUARD,), 0x5A, dtype=torch.uint8, device="cuda")
    buf[GUARD:GUARD + size] = 0
    for _ in range(2):  # the second pass runs on the tickets and records that the first one left
        tokens = tokens0.clone()
        counts, flags = outputs(n_seq)
        wino.wino_step(H, Wd, tokens, p, counts, buf[GUARD:GUARD + size], flags=flags)
    torch.cuda.synchronize()
    assert torch.all(buf[:GUARD] == 0x5A) and torch.all(buf[GUARD + size:] == 0x5A), "written outside the workspace"
    assert wino.wino_read_device_status(buf[GUARD:GUARD + size]) == wino.WINO_OK

    # the same sequences as a batch of their own, in a workspace with room to spare
    idx = torch.arange(n_seq, device="cuda") if listed is None else act.long()
    rows = w.kinds * L
    H_sub = H.view(n_seq, rows, w.d)[idx].reshape(-1, w.d).contiguous()
    ref = tokens0[idx].contiguous()
    counts_ref, flags_ref = outputs(len(idx))
    q = params(len(idx))
    wino.wino_step(H_sub, Wd, ref, q, counts_ref,
                   torch.zeros(wino.wino_workspace_size_step(q, w.d, w.V) + 4 * GUARD, dtype=torch.uint8, device="cuda"),
                   flags=flags_ref)
    torch.cuda.synchronize()
    assert torch.equal(tokens[idx], ref) and torch.equal(counts[idx], counts_ref) and torch.equal(flags[idx], flags_ref)
    assert torch.any(ref != tokens0[idx]), "the step changes something"
    rest = torch.ones(n_seq, dtype=torch.bool, device="cuda")
    rest[idx] = False
    assert torch.equal(tokens[rest], tokens0[rest])
    assert torch.all(counts[rest] == -9) and torch.all(flags[rest] == -9)
