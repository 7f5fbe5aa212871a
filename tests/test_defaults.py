"""What plans start with, decided without a GPU (fake_gpu.py): float sums keep
the grouping that the sub-band kernels give them, and the time model orders
setups whose fastest variants are known from timings."""
import numpy as np
import pytest

from fake_gpu import probe

SUBBANDS = (2, 3, 4, 6)


def grouped(v):
    """Whether a variant sums groups of four channels before it accumulates."""
    kind, dpt, spt = v[:3]
    return kind in SUBBANDS or (kind == 0 and (dpt * spt == 8 or (dpt, spt) == (4, 8)))


# Setups whose channel groups share few delay patterns, so that a sub-band
# variant fits them: few and many trials, few and many channels.
GROUPED = [
    ("apertif", 1, 1024, 16, 20000, "f32"), ("apertif", 2, 1024, 8, 20000, "f16"),
    ("wide", 4, 512, 20, 8192, "f32"), ("wide", 16, 300, 4, 8192, "bf16"),
    ("lband", 384, 64, 4, 4096, "f32"), ("lband", 303, 40, 7, 1934, "f32"),
    ("lband", 72, 88, 7, 5162, "bf16"), ("lband", 7, 80, 37, 8030, "f32"),
    ("lband", 99, 92, 27, 5988, "f32"), ("lband", 238, 72, 22, 3260, "f32"),
    ("lband", 247, 120, 67, 1347, "f32"), ("wide", 8, 219, 101, 9289, "f32"),
    ("apertif", 1, 1024, 2048, 20000, "f32"), ("wide", 2, 509, 777, 10001, "f16"),
]
# No sub-band variant fits these; one chain over the channels is all they ever had.
FREE = [("lband", 96, 64, 64, 4096, "f32"), ("lofar", 1, 32, 2048, 200000, "f32")]


@pytest.fixture(scope="module")
def answers(tmp_path_factory):
    req = [{"setups": [s], "ask": ["adjoint"] if s[5] == "f32" else []} for s in GROUPED + FREE]
    return dict(zip(GROUPED + FREE, probe(req, tmp_path_factory.mktemp("fake"))))


@pytest.mark.parametrize("setup", GROUPED, ids=str)
def test_float_sums_keep_their_channel_groups(answers, setup):
    assert grouped(answers[setup]["plans"][0]), answers[setup]


@pytest.mark.parametrize("setup", [s for s in GROUPED if s[5] == "f32" and s[2] > 128], ids=str)
def test_adjoint_sums_keep_their_groups(answers, setup):
    """The transposed plan sums over trials; at these bands its groups of four
    trials share few patterns too."""
    assert grouped(answers[setup]["adjoint"]), answers[setup]


def test_plans_without_sub_bands_may_chain(answers):
    assert [answers[s]["plans"][0][:3] for s in FREE] == [[5, 4, 22], [0, 8, 8]]


# (setup, starting keys that timings on a GB300 bear out, launch order)
SMALL = [[0, 2, 4], [0, 4, 2]]
KNOWN = [
    (("apertif", 1, 1024, 2048, 20000, "f32"), [[6, 4, 8]], 0),
    (("apertif", 1, 1024, 2048, 20000, "u8"), [[4, 4, 8]], 0),
    (("lband", 96, 64, 64, 4096, "f32"), [[5, 4, 22]], 0),
    (("lband", 96, 64, 64, 4096, "u8"), [[0, 4, 20]], 0),
    (("lofar", 1, 32, 2048, 200000, "f32"), [[0, 8, 8]], 1),
    # two partial-sum slots of 32 channels do not fit, one does (203 against 225 us)
    (("apertif", 1, 439, 287, 19105, "f16"), [[6, 4, 8]], 0),
    (("wide", 2, 509, 777, 10001, "f16"), [[4, 4, 8]], 0),
    # one beam, few trials: small tiles (18 to 27 us) against sub-bands (44)
    (("wide", 1, 281, 128, 2189, "f32"), SMALL, 0),
    (("wide", 1, 150, 67, 2091, "f32"), SMALL, 0),
    (("wide", 1, 223, 86, 2534, "bf16"), SMALL, 0),
]


def test_known_fastest_variants(tmp_path):
    got = probe([{"setups": [s]} for s, _, _ in KNOWN], tmp_path)
    for a, (setup, keys, order) in zip(got, KNOWN):
        assert a["plans"][0][:3] in keys and a["orders"][0] == order, (setup, a)


LBAND96 = ("lband", 96, 64, 64, 4096)
WIDE4 = ("wide", 4, 512, 1000, 8192)
LOWFREQ = ("lowfreq", 4, 208, 500, 4000)


@pytest.fixture(scope="module")
def batches(tmp_path_factory):
    pairs = {"free + grouped": [LBAND96, WIDE4], "grouped + free": [WIDE4, LBAND96],
             "grouped + free 2": [("lband", 43, 46, 17, 2000), LOWFREQ],
             "free": [LBAND96, LOWFREQ]}
    req = {(n, t): {"setups": [list(s) + [t] for s in p], "ask": ["batch"]}
           for n, p in pairs.items() for t in ("f32", "f16", "u8")}
    req["chosen"] = {"setups": [list(LBAND96) + ["f32"], list(WIDE4) + ["f32"]], "ask": ["batch"],
                     "set": [5, 4, 14, 4, 1, 8, 3]}
    return dict(zip(req, probe(list(req.values()), tmp_path_factory.mktemp("fake"))))


@pytest.mark.parametrize("pair", ["free + grouped", "grouped + free", "grouped + free 2"])
@pytest.mark.parametrize("dtype", ["f32", "f16"])
def test_batches_keep_the_groups_of_every_plan(batches, pair, dtype):
    """A float plan that keeps its channel groups alone keeps them in a batch,
    whatever stands beside it."""
    assert grouped(batches[pair, dtype]["batch"]), batches[pair, dtype]


def test_batches_with_other_rules(batches):
    """8-bit sums in any order, and the first plan's variant where the caller
    set one."""
    assert batches["free", "u8"]["batch"][:3] == [0, 4, 20]
    assert batches["chosen"]["batch"] == [5, 4, 14, 4, 1, 8, 3]


@pytest.mark.parametrize("order", [0, 1])
def test_adjoint_keeps_its_launch_order(tmp_path, order):
    """The adjoint's plan starts in the launch order that goes with its
    variant (here a tuning cache's), and its launch uses that order."""
    setup = ("lofar", 1, 8, 16, 3000, "f32")
    v = [0, 4, 4, 2, 2, 4, 3]
    got = probe([{"setups": [setup], "transposed": v + [order], "ask": ["adjoint"]}], tmp_path)[0]
    args = [x["args"] for x in got["adjoint_launches"] if "args" in x]
    assert len(args) == 1 and (args[0]["C"], args[0]["D"]) == (16, 8)
    assert got["adjoint"] == v and args[0]["time_major"] == order, got


@pytest.mark.parametrize("setup,least", [(("lofar", 1, 32, 2048, 200000, "f32"), 1000),
                                         (("lofar", 1, 16, 64, 1000, "u8"), 16),
                                         (("wide", 1, 512, 1024, 4096, "bf16"), 512)], ids=str)
def test_stream_fill_covers_the_machine(tmp_path, setup, least):
    """A push with few long rows fills its buffer with several blocks per row
    (152 SMs), one with many short rows with one per row."""
    fill = probe([{"setups": [setup], "ask": ["stream"]}], tmp_path)[0]["stream_launches"][0]
    assert fill["smem"] == 0 and fill["grid"][0] == setup[1] * setup[2]
    assert least <= fill["grid"][0] * fill["grid"][1] <= max(least, 16 * 152), fill


def test_tuner_times_candidates_in_their_own_order(tmp_path):
    """A default that is fast only with time tiles fastest is not given up for
    a slower variant."""
    got = probe([{"setups": [("lofar", 1, 32, 64, 100000, "f32")], "ask": ["tune"]}], tmp_path)[0]
    assert got["orders"] == [1], got
    v, order, best, ms = got["tuned"]
    assert order == 1 and best == v and ms == 0.5 and v[:5] == got["plans"][0][:5], got


def test_batches_take_the_longest_tiles_first(tmp_path):
    """All plans of a batch run tiles of one shape: those with the most channels
    come first, whatever tiles the plans take on their own."""
    setups = [["lband", 96, 64, 64, 4096, "u8"], ["lband", 1, 100, 20, 1000, "u8"],
              ["lowfreq", 4, 208, 500, 4000, "u8"]]
    got = probe([{"setups": setups, "ask": ["batch"]}, {"setups": setups[:2], "ask": ["batch"]}],
                tmp_path)
    assert [g["batch_channels"] for g in got] == [[208, 100, 64], [100, 64]]


def test_refusals_name_what_is_accepted(tmp_path):
    """Chunks of 1 and 2 channels exist for the wide kernels only; the refusal
    of another size says so."""
    bad = [[0, 8, 8, 1, 8, 3, 3], [0, 4, 8, 4, 1, 2, 3]]
    for a in probe([{"setups": [list(LBAND96) + ["f32"]], "refuse": v} for v in bad], tmp_path):
        assert "4, 8, 16 or 32" in a["message"] and "1 and 2" in a["message"], a


@pytest.mark.parametrize("setup", [("lowfreq", 5, 95, 220, 2494, "f32"),
                                   ("lowfreq", 6, 74, 121, 2801, "f32"),
                                   ("lowfreq", 3, 111, 266, 5410, "f32")], ids=str)
def test_adjoint_windows_are_sized_by_the_widest_steps(tmp_path, setup):
    """A transposed table steps unevenly: tiles of 8 trials x 512 samples, which
    the mean step lets two blocks per SM hold, are 1.7 times slower there than
    4 x 1024 (165 us against 276 for the first)."""
    got = probe([{"setups": [setup], "ask": ["adjoint"]}], tmp_path)[0]
    assert got["adjoint"][:5] == [0, 4, 8, 1, 4] or got["adjoint"][:5] == [0, 4, 8, 1, 8], got


def test_group_rule_equals_the_built_tables(tmp_path):
    """The quick look at a delay table says what building the list's sub-band
    variants says: Eq. 1 tables, equal patterns with wide spans (shared memory
    decides), steps in stairs, no order, a single step for all channels."""
    rng = np.random.default_rng(3)
    tables = []
    for i in range(200):
        C, D, mode = int(rng.integers(1, 70)), int(rng.integers(1, 200)), i % 5
        if mode == 0:
            f = rng.uniform(100, 1500) * (1 + np.arange(C) * rng.uniform(0.01, 0.3) / C)
            d = np.arange(D) * rng.uniform(0.01, 2) * 4.148808e3 / 10 ** rng.uniform(-5.3, -3.5)
            sh = np.floor(d[:, None] * (f ** -2.0 - f[-1] ** -2.0) + 0.5)
        elif mode == 1:
            sh = np.sort(rng.integers(0, rng.integers(1, 2000), (D, C)), axis=0)
        elif mode == 2:
            sh = rng.integers(0, rng.integers(1, 4000), (D, 1)) + rng.integers(0, 2, (1, C))
        elif mode == 3:
            sh = ((np.arange(D) // rng.integers(1, 8) * rng.integers(1, 300))[:, None]
                  + rng.integers(0, rng.integers(1, 3000), (1, C)))
        else:
            sh = np.arange(D)[:, None] * rng.integers(0, 400) + np.zeros((1, C))
        tables.append([np.minimum(sh, 1 << 26).astype(int).tolist(), int(rng.integers(1, 3000)),
                       ["f32", "f16"][i % 2]])
    got = probe([{"tables": tables}], tmp_path)[0]
    assert 40 <= sum(f for f, _ in got) <= 160
    assert [i for i, (f, k) in enumerate(got) if f != k] == []
