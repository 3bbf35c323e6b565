"""Tile launches are cut into units (parts of few long tiles, runs of many short ones with
adjacent tiles joined, units taken over by running blocks).  Whatever the cut, each call over
TILES equals, bit for bit, the same call over the INDICES list of the same elements, whose
kernels know no units and are checked against the oracle elsewhere."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

SEEDS = (11, 2**40 + 5)


@pytest.fixture(scope="module")
def copes():
    from paper_2608_02391_gb300 import copes as c
    c.load()
    return c


def arena(copes, n, dtype):
    gen = torch.Generator("cuda").manual_seed(n)
    master = torch.randn(n, generator=gen, device="cuda") * 0.02
    return copes.Arena(torch.zeros(n, dtype=dtype, device="cuda"), master,
                       *[torch.zeros(n, dtype=dtype, device="cuda") for _ in range(3)])


def index_list(copes, ranges):
    idx = torch.cat([torch.arange(b, e, device="cuda") for b, e in ranges])
    return copes.SubspaceHandle(copes.SUBSPACE_INDICES, idx, idx.numel())


def steps(copes, a, sub, pairs):
    """Every tile kernel once; two pairs as two pair calls where sub takes none."""
    out = []
    copes.init_normal(a, sub, 7, 0.5, 0.02)
    out += [a.master.clone(), a.w3.clone()]
    copes.perturb(a, sub, SEEDS[0], 1e-3)
    out.append(a.w.clone())
    if pairs:
        copes.perturb_two_pairs(a, sub, *SEEDS, 1e-3)
        out += [c.clone() for c in a.copies]
    else:
        for seed in SEEDS:
            copes.perturb_pair(a, sub, seed, 1e-3, a.w2)
            out += [a.w.clone(), a.w2.clone()]
    copes.perturb_pair(a, sub, SEEDS[1], -2e-3, a.w2)
    out += [a.w.clone(), a.w2.clone()]
    copes.perturb_partner(a, sub, a.w2)
    out.append(a.w.clone())
    copes.restore(a, sub)
    out += [c.clone() for c in a.copies]
    nid, sign, P = copes.member_table(6, copes.ANTITHETIC)
    f = torch.tensor([1.0, -0.5, 0.25, 2.0, -1.5, 0.75], device="cuda")
    copes.update(a, sub, nid, sign, f, copes.member_seeds(33, 1, 2, P), 1e-2)
    out += [a.master] + a.copies
    copes.check()
    return out


CASES = [
    # few tiles, cut into parts: aligned, cut at odd places, shorter than a part, very long
    (60_000, [(0, 49_152)], 16_384), (60_001, [(3, 16_390), (20_000, 60_001)], 16_384),
    (200_000, [(64, 200_000)], 65_536), (3_000_000, [(1, 1_048_577), (1_500_002, 2_999_999)], 1 << 20),
    (40_000, [(5, 7), (9, 10), (4_096, 8_193)], 16_384), (50_000, [(7, 49_999)], 300),
    # units of exactly one part, and tiles on both sides of the counts at which the cut changes
    (4096 * 499, [(0, 4096 * 499)], 4_096), (4096 * 501 + 5, [(0, 4096 * 501 + 5)], 4_096),
    (16_384 * 607, [(0, 16_384 * 607)], 16_384), (16_384 * 609 + 1, [(0, 16_384 * 609 + 1)], 16_384),
    # short tiles in runs: joined, with gaps between ranges, single elements
    (120_000, [(0, 120_000)], 100), (130_000, [(k * 130 + k % 3, k * 130 + 97) for k in range(1000)], 32),
    (70_000, [(1, 69_999)], 16), (6_000, [(2 * k, 2 * k + 1) for k in range(3000)], 4),
    # a third of the arena: shorter tiles than the bound says
    (5_000_000, [(3_300_001, 4_966_668)], 1000),
    # runs of eight tiles, about two waves of units
    (2048 * 8000, [(2, 2048 * 8000)], 2_048),
    # runs with more than three waves of units, taken over early and late: aligned tiles joined to
    # default ones (the noise ops' units), and odd ones with gaps between them (the update's)
    (4096 * 8000, [(0, 4096 * 8000)], 4_096),
    (33_000_000, [(k * 3_300_000 + k, (k + 1) * 3_300_000 - 5_000) for k in range(10)], 1_000),
]
EARLY_RUNS = {16: "perturb", 17: "update"}


@pytest.mark.parametrize("case", range(len(CASES)))
def test_every_cut_equals_the_index_list(copes, case):
    n, ranges, tile = CASES[case]
    for dtype in (torch.bfloat16, torch.float32):
        got = steps(copes, arena(copes, n, dtype), copes.tiles_from_ranges(ranges, tile_size=tile), True)
        want = steps(copes, arena(copes, n, dtype), index_list(copes, ranges), False)
        # two pairs: w, w2 of the first pair, w3, w4 of the second
        for i, (x, y) in enumerate(zip(got, want)):
            assert torch.equal(x, y), f"output {i}, {dtype}"


def test_invalid_tile_in_a_run_is_left_out(copes):
    n, tile = 64_000, 32
    a = arena(copes, n, torch.bfloat16)
    sub = copes.tiles_from_ranges([(0, n)], tile_size=tile)
    bad = [0, 7, 8, 31, 32, 1999]
    sub.tensor[bad, 1] = n + 1  # past the arena's end
    copes.perturb(a, sub, SEEDS[0], 1e-3)
    with pytest.raises(copes.CopesError) as e:
        copes.check()
    assert e.value.code == copes.ERR_DEVICE_CHECK and "0x1:" in str(e.value)
    b = arena(copes, n, torch.bfloat16)
    copes.perturb(b, copes.tiles_from_ranges([(0, n)], tile_size=tile), SEEDS[0], 1e-3)
    want = b.w.clone()
    for t in bad:
        want[t * tile:(t + 1) * tile] = 0
    assert torch.equal(a.w, want)


@pytest.mark.parametrize("size", [4096, 16_384])
def test_reversed_tile_is_left_out(copes, size):
    """A tile with b > e whose e - b wraps round to a whole part or tile."""
    n = 4 * size
    sub = copes.tiles_from_ranges([(0, n)], tile_size=size)
    sub.tensor[1] = torch.tensor([-size, 0], device="cuda")  # [2^64 - size, 0)
    a, b = arena(copes, n, torch.bfloat16), arena(copes, n, torch.bfloat16)
    rest = index_list(copes, [(0, size), (2 * size, n)])
    for x, s in ((a, sub), (b, rest)):
        copes.perturb_pair(x, s, SEEDS[0], 1e-3, x.w2)
    copes.restore(a, sub)
    copes.restore(b, rest)
    with pytest.raises(copes.CopesError) as e:
        copes.check()
    assert e.value.code == copes.ERR_DEVICE_CHECK and "0x1:" in str(e.value)
    assert torch.equal(a.master, b.master) and all(torch.equal(x, y) for x, y in zip(a.copies, b.copies))


@pytest.mark.parametrize("offset", [0, 4])  # floats before theta: 32-byte aligned or not
@pytest.mark.parametrize("begin", [0, 4, 8, 3])
def test_two_pairs_over_whole_tiles_equal_pairs(copes, begin, offset):
    """Enough default tiles to stay whole: by octets where theta's addresses allow them."""
    n = begin + 1300 * 16_384 + 5
    master = (torch.randn(n + offset, device="cuda") * 0.02)[offset:]
    a = copes.Arena(torch.zeros(n, dtype=torch.bfloat16, device="cuda"), master,
                    *[torch.zeros(n, dtype=torch.bfloat16, device="cuda") for _ in range(3)])
    sub = copes.tiles_from_ranges([(begin, n)], tile_size=16_384)
    copes.perturb_two_pairs(a, sub, *SEEDS, 1e-3)
    got = [c.clone() for c in a.copies]
    for k, seed in enumerate(SEEDS):
        a.w.zero_(), a.w2.zero_()
        copes.perturb_pair(a, sub, seed, 1e-3, a.w2)
        assert torch.equal(a.w, got[2 * k]) and torch.equal(a.w2, got[2 * k + 1])
    copes.check()


@pytest.mark.parametrize("tiles", [130, 187, 679, 1217, 1860])
@pytest.mark.parametrize("P", [4, 8, 9, 40])
def test_update_cuts_equal_the_index_list(copes, P, tiles):
    """Tile counts and noise vectors at which the update's tiles are cut differently, and on both
    sides of the count up to which theta is asked for ahead."""
    begin, size = 6, 9_000  # longer than half the default tile, so that tiles are not joined
    n = begin + tiles * size - 777
    nid, sign, _ = copes.member_table(2 * P, copes.ANTITHETIC)
    f = torch.linspace(-1, 1, 2 * P, device="cuda")
    got = []
    for sub in (copes.tiles_from_ranges([(begin, n)], tile_size=size), index_list(copes, [(begin, n)])):
        a = arena(copes, n, torch.bfloat16)
        copes.update(a, sub, nid, sign, f, copes.member_seeds(33, 1, 2, P), 1e-2)
        got.append([a.master] + a.copies)
    for x, y in zip(*got):
        assert torch.equal(x, y)
    copes.check()
