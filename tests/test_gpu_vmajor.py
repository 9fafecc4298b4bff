"""The vocabulary-major score kernel (csrc/score_vmajor.cu) against the fp64 oracle, at the edges of its row counts:
one row, partial 32-row chunks, one accumulator of 32-multiple and of 16-multiple width, two accumulators of unequal
and of equal width, several row groups with a ragged last one; vocabulary and K tails; with and without entropy.
The launch's timeline shows its tiles, and wino_score_launch that this kernel takes it (the tile counts of the first three
shapes are those of the row-block split too, the others' are not)."""
import math

import numpy as np
import pytest
import torch

import oracle
import wino_synth as ws

pytestmark = pytest.mark.gpu

# (N, d, V, tiles of the launch: row groups x vocabulary tiles)
SHAPES = [
    (1, 8, 19456, 1 * 76),         # one row, one K slice (mostly zero fill), one 32-column chunk
    (33, 72, 20001, 1 * 139),      # 64 columns, K tail, 144-wide tiles, the last one mostly past the vocabulary
    (48, 256, 40000, 1 * 228),     # 176-wide tiles
    (40, 136, 47502, 1 * 213),     # 224-wide tiles
    (257, 512, 19456, 2 * 76),     # two groups of one accumulator of 144 columns (a half chunk at its end)
    (392, 512, 19456, 2 * 76),     # 208 columns
    (482, 512, 19456, 2 * 76),     # 256 columns
    (257, 1024, 19456, 1 * 76),    # 144 + 128 columns, three accumulators in TMEM
    (327, 1544, 29557, 1 * 116),   # 176 + 160 columns, two accumulators in TMEM, K and vocabulary tails
    (518, 1024, 19456, 2 * 76),    # two groups of 144 + 128 columns, the second ragged
    (257, 2056, 19457, 1 * 77),    # a last tile of one entry whose two accumulators go to two pairs
    (536, 2048, 20233, 2 * 80),    # two groups, 4 last tiles shared by 8 of each group's 38 pairs
    (726, 1024, 24118, 3 * 95),    # three groups
]


def _tiles(H, W, N, d, V):
    """Tiles computed by one launch, from its timeline."""
    import paper_2605_16941_gb300 as wino
    buf = torch.zeros(256 * wino.TIMELINE_WORDS, dtype=torch.int64, device="cuda")
    out = [torch.empty(N, dtype=t, device="cuda") for t in (torch.int32, torch.float32, torch.float32)]
    wsp = wino.workspace(N, d, V)
    torch.cuda.synchronize()
    wino.wino_timeline_begin(buf, 1, 256)
    try:
        wino.wino_score_rows(H, W, None, *out, wsp, N=N, d=d, V=V)
        torch.cuda.synchronize()
    finally:
        wino.wino_timeline_end()
    T = buf.view(256, wino.TIMELINE_WORDS).cpu().numpy().view(np.uint64)
    return int((T[0::2, 7] & np.uint64(0xFFFFFFFF)).sum())


@pytest.mark.parametrize("N,d,V,tiles", SHAPES, ids=[f"N{s[0]}_d{s[1]}_V{s[2]}" for s in SHAPES])
def test_matches_oracle(N, d, V, tiles):
    import paper_2605_16941_gb300 as wino
    from gpu_helpers import compare_rows, dev, gpu_score
    plan = wino.wino_score_launch(N, d, V)
    assert plan["kernel"] == 2 and plan["n_groups"] * plan["n_vt"] == tiles
    H = ws.random_bf16(N, d, 1.0, seed=N * 5 + d)
    W = ws.random_bf16(V, d, 1.0 / math.sqrt(d), seed=V + d)
    rng = np.random.default_rng(N + V)
    target = rng.integers(-1, V, size=N).astype(np.int32)
    target[: min(N, 3)] = [V - 1, 0, V // 2][: min(N, 3)]
    W[target[0]] = H[0]  # a certain row whose winner is the last vocabulary entry
    Hd, Wd = dev(H), dev(W)
    assert _tiles(Hd, Wd, N, d, V) == tiles
    o = oracle.score_rows(H, W, target)
    for entropy in (False, True):
        compare_rows(o, gpu_score(Hd, Wd, target, entropy=entropy))


def test_exact_ties_pick_lowest_index():
    """Equal logits in different lane quarters, CTAs and tiles: the smallest vocabulary id wins."""
    from gpu_helpers import dev, gpu_score
    N, d, V = 40, 64, 20000
    H = ws.random_bf16(N, d, 1.0, seed=6)
    W = ws.random_bf16(V, d, 0.05, seed=5)
    H[0] = ws.f32_to_bf16_bits(np.random.default_rng(9).integers(-4, 5, size=d).astype(np.float32))
    H[1] = 0  # every logit 0: argmax must be 0
    for v in (19999, 12345, 300, 77, 45):
        W[v] = H[0]
    g = gpu_score(dev(H), dev(W), None)
    assert g.argmax[0] == 45 and g.argmax[1] == 0
    assert abs(g.pmax[1] - 1.0 / V) < 1e-8
