"""Which score kernel a launch gets (wino_score_launch) and the vocabulary-major kernel's work split, on the CPU: every
(row group, vocabulary tile, accumulator) goes to exactly one CTA pair, the rows of the groups cover N, the accumulators
fit tensor memory, the records fit the workspace, the ring fits shared memory and keeps one CTA per SM, and the
measured shapes run on the kernel that they were measured on."""
import itertools
import math

import pytest

import paper_2605_16941_gb300 as wino

SMEM_MAX = 227 * 1024  # dynamic shared memory a CTA may request
SM_SHARED = 228 * 1024  # shared memory of one SM
OVERHEAD = 1024 + 512 + 8 * 4096  # ring alignment slack + barrier block + transposes

DEVICES = [(152, 76), (148, 74), (132, 66), (8, 4), (2, 1)]
ROWS = [1, 16, 32, 33, 48, 49, 64, 96, 128, 129, 208, 255, 256, 257, 288, 300, 320, 333, 352, 400, 511, 512, 513, 726, 768,
        1000, 1024, 1025, 1298, 1664, 2048, 2049, 4096, 1 << 24]
DIMS = [8, 64, 256, 320, 512, 1024, 1536, 4096, 65536]
VOCABS = [2, 1000, 19455, 19456, 20001, 32000, 100003, 126464, 134400, 1 << 27]


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2605_16941_gb300 import build
    build.build()


def _work(p):
    """(group, tile, accumulator) -> pairs that compute it, as the kernel's three roles walk their items."""
    own = {}
    full, rem = divmod(p["n_vt"], p["G"])
    accs = 2 if p["hw1"] else 1
    for c in range(p["ctas"] // 2):
        grp, col = c % p["n_groups"], c // p["n_groups"]
        for i in itertools.count():
            half = p["split"] and i == full
            vt = i * p["G"] + (col // 2 if half else col)
            if not (col < 2 * rem if half else vt < p["n_vt"]):
                break
            for h in ([col % 2] if half else range(accs)):
                own.setdefault((grp, vt, h), []).append(c)
    return own, accs


@pytest.mark.parametrize("sm,pairs", DEVICES, ids=[f"sm{a}_p{b}" for a, b in DEVICES])
def test_split_invariants(sm, pairs):
    units = min(pairs, sm // 2)
    kernels = set()
    for N, d, V in itertools.product(ROWS, DIMS, VOCABS):
        p = wino.wino_score_launch(N, d, V, sm, pairs)
        kernels.add(p["kernel"])
        assert p["smem_bytes"] <= SMEM_MAX and 2 * p["smem_bytes"] > SM_SHARED, p  # one TMEM owner per SM
        assert p["n_groups"] * p["G"] <= units and p["ctas"] == 2 * p["n_groups"] * p["G"], p
        assert p["n_vt"] == math.ceil(V / p["bn"]) and p["bn"] % 16 == 0 and 128 <= p["bn"] <= 256, p
        assert p["records"] <= min(math.ceil(V / 128), 256), p
        assert wino.wino_workspace_size(N, d, V) >= N * p["records"] * 16
        if p["kernel"] != 2:
            row = wino.wino_score_plan_host(N, d, V, sm, pairs)
            assert p["kernel"] == row["two"] and p["records"] == row["G"]
            assert all(p[k] == row[k] for k in ("bn", "n_vt", "n_groups", "G", "ctas", "stages", "stage_bytes"))
            assert p["hw0"] == p["hw1"] == p["slots"] == p["split"] == 0
            continue
        hw0, hw1 = p["hw0"], p["hw1"]
        rows = hw0 + hw1
        # 8-row swizzle atoms: each CTA stages half of an accumulator's rows
        assert hw0 % 16 == 0 and hw1 % 16 == 0 and 32 <= hw0 <= 256 and 0 <= hw1 <= hw0 and rows // 2 <= 256, p
        assert rows * p["n_groups"] >= N > rows * (p["n_groups"] - 1), p
        # every accumulator, read in whole 32-column chunks, lies in the 512 columns of tensor memory
        accs = 2 if hw1 else 1
        assert max(2, accs) <= p["slots"] <= 4, p
        for hw in (hw0, hw1):
            assert (p["slots"] - 1) * hw0 + math.ceil(hw / 32) * 32 <= 512, p
        assert p["records"] == 2 * p["G"], p
        assert p["stage_bytes"] == 16384 + rows // 2 * 128 and p["stage_bytes"] % 1024 == 0, p
        ring = p["stages"] * p["stage_bytes"]
        assert 2 <= p["stages"] <= 12 and p["smem_bytes"] == ring + OVERHEAD, p
        assert ring >= 512 * 4 * 20, p  # the row states of the four lane quarters at the end
        assert not p["split"] or (hw1 and 0 < 2 * (p["n_vt"] % p["G"]) <= p["G"]), p
    assert kernels == ({0, 1, 2} if units > 1 else kernels)


@pytest.mark.parametrize("N,d,V", [(1, 8, 19456), (33, 72, 20001), (64, 4096, 126464), (257, 512, 19456), (300, 4096, 126464),
                                   (333, 1024, 32000), (352, 4096, 126464), (257, 2056, 19457), (536, 2048, 20233),
                                   (726, 1024, 24118), (1000, 1536, 100003), (1024, 4096, 126464)])
def test_every_accumulator_once(N, d, V):
    p = wino.wino_score_launch(N, d, V, 152, 76)
    assert p["kernel"] == 2, p
    own, accs = _work(p)
    assert sorted(own) == sorted(itertools.product(range(p["n_groups"]), range(p["n_vt"]), range(accs)))
    assert all(len(v) == 1 for v in own.values())
    assert all(v[0] % p["n_groups"] == g for (g, _, _), v in own.items())


def test_measured_shapes():
    """The kernel and split of the measured steps on a GB300 (152 SMs, 76 resident pairs)."""
    def launch(N, d=4096, V=126464):
        p = wino.wino_score_launch(N, d, V, 152, 76)
        return tuple(p[k] for k in ("kernel", "n_groups", "hw0", "hw1", "bn"))
    assert launch(64) == (2, 1, 64, 0, 240)
    assert launch(128) == (2, 1, 128, 0, 240)
    assert launch(256)[0] == 0 and launch(2048, V=134400)[0] == 1 and launch(64, 64, 1000)[0] == 0
    assert launch(300) == (2, 1, 160, 144, 256)
    assert launch(352) == (2, 1, 176, 176, 256)
    assert launch(1024) == (2, 4, 256, 0, 256)
    assert launch(1000, 1536, 100003)[0] == 2 and launch(333, 1024, 32000)[0] == 2


def test_launch_argument_errors():
    for args in ((256, 4096, 126464, 1, 76), (256, 4096, 126464, 152, 0), (256, 4096, 126464, 0, 76), (0, 4096, 126464, 152, 76),
                 (256, 60, 126464, 152, 76)):
        with pytest.raises(wino.WinoError):
            wino.wino_score_launch(*args)
