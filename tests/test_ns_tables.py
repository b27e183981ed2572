"""The work tables that persistent launches claim from, as they run: merged
iterations (3 to 8 iterations of wide frames), launches that mix them with
iterated frames, and 128-wide tiles.  tests/test_ns_schedule.py covers the
iterated form in 256-wide tiles; here the same properties hold for every table
that a step takes:
  * every matrix runs its own form's products in order, each tile of each
    product exactly once;
  * an item waits exactly for the previous product of its own matrix, complete;
  * when an item is claimed, every item it waits for was claimed before it
    (claims happen only in running CTAs, so this makes the schedule deadlock-free).
What is expected is written out here, not taken from the library."""
import numpy as np
import pytest

from paper_2608_05088_gb300 import build, inputs

SIGNALS_PER_ITEM = 16   # epilogue warps of a CTA pair
GRAM, PP, BX = 0, 1, 2
# a Gram product, the p x p products of the merged iterations, a product with X
GROUP = {1: [GRAM, PP, BX], 2: [GRAM] + [PP] * 5 + [BX], 3: [GRAM] + [PP] * 9 + [BX]}
GROUPS = {3: [2], 4: [2, 1], 5: [2, 2], 6: [2, 2, 1], 7: [2, 2, 2], 8: [2, 2, 3]}


@pytest.fixture(scope="module")
def malt():
    build.build()
    import paper_2608_05088_gb300.malt as m
    return m


def cdiv(a, b):
    return -(-a // b)


def kinds(k, grouped):
    if not grouped:
        return [GRAM, PP, BX] * k
    return sum([GROUP[g] for g in GROUPS[k]], [GRAM, PP, BX])


def tiles(frame, kind, width):
    p, q = frame
    if kind == BX:
        return cdiv(p, 256) * cdiv(q, width)
    # a row of 256-high tiles starts at the diagonal
    return sum(cdiv(p, width) - r * (256 // width) for r in range(cdiv(p, 256)))


def check(tab, shapes, k, grouped, width):
    """grouped: which matrices run merged iterations."""
    n = len(shapes)
    frames = [tuple(sorted((cdiv(a, 8) * 8, cdiv(b, 8) * 8))) for a, b in shapes]
    want = [kinds(k, g) for g in grouped]
    assert set(tab[:, 8].tolist()) == {width}
    order = {}
    slots = {}
    for grp in np.unique(tab[:, 0]):
        done = {}
        for _, st, kind, mat, local, dep, target, items, _, cls, b in tab[tab[:, 0] == grp].tolist():
            assert kind == want[mat][st]
            assert items == tiles(frames[mat], kind, width)
            assert slots.setdefault((grp, cls, b), mat) == mat
            if st == 0:
                assert dep == -1 and target == 0
            else:
                prev = tiles(frames[mat], want[mat][st - 1], width)
                assert dep == (st - 1) * n + mat and target == SIGNALS_PER_ITEM * prev
                # claimed in order with every item finishing at once
                assert done[mat, st - 1] == target
            done[mat, st] = done.get((mat, st), 0) + SIGNALS_PER_ITEM
            order.setdefault((mat, st), []).append(local)
    assert set(order) == {(i, s) for i in range(n) for s in range(len(want[i]))}
    for (mat, st), locs in order.items():
        assert sorted(locs) == list(range(tiles(frames[mat], want[mat][st], width))), (mat, st)
    # a slot of a class holds one matrix and every class one frame
    assert len(slots) == len(set(slots.values())) == n
    of_class = {}
    for (grp, cls, _), mat in slots.items():
        assert of_class.setdefault((grp, cls), frames[mat]) == frames[mat]


@pytest.mark.parametrize("k", [1, 2, 3, 4, 5, 6, 7, 8, 9, 64])
@pytest.mark.parametrize("muon", [False, True])
def test_gpt2_small_mixes_both_forms(malt, k, muon):
    """768 x 2304 and 768 x 3072 (both ways) merge iterations, 768 x 768 does not."""
    shapes = list(inputs.first_layers(inputs.WORKLOADS["gpt2_small"], 12 if k < 9 else 3).shapes)
    merges = (4 if muon else 3) <= k <= 8
    # (3 layers: 72 symmetric tiles, still wide)
    check(malt.malt_ns_tables(shapes, malt.hparams(ns_steps=k), muon), shapes, k,
          [merges and max(s) >= 2 * min(s) for s in shapes], 256)


@pytest.mark.parametrize("k", [3, 5, 8])
def test_narrow_tiles(malt, k):
    """Few tiles: 128 columns wide; frames with ragged last tiles, both forms."""
    shapes = [(256, 4096), (2184, 264), (136, 136), (8, 8), (520, 392), (77, 300), (264, 4000)]
    grouped = [True, True, False, False, False, False, True]
    check(malt.malt_ns_tables(shapes, malt.hparams(ns_steps=k)), shapes, k, grouped, 128)


@pytest.mark.parametrize("shapes,grouped", [
    ([(776, 1560)] * 5 + [(1560, 776)] * 4 + [(776, 776)], [True] * 9 + [False]),
    # ten frames: two launches, the shorter reductions in the second, iterated only
    ([(256, 512 * (i + 9)) for i in range(8)] + [(256, 256), (520, 520)] * 12, [True] * 8 + [False] * 24),
])
def test_ragged_wide_tiles_and_two_launches(malt, shapes, grouped):
    for k in (3, 5, 8):
        check(malt.malt_ns_tables(shapes, malt.hparams(ns_steps=k)), shapes, k, grouped, 256)


def test_coefficients_outside_the_rule(malt):
    shapes = [(256, 4096), (2184, 264)]
    hp = malt.hparams(ns_coeffs=(10.0, -4.0, 1.0))
    check(malt.malt_ns_tables(shapes, hp), shapes, 5, [False, False], 128)


def test_bad_arguments(malt):
    for shapes, hp in (([(256, 512)], malt.hparams(ns_steps=0)), ([(256, 512)], malt.hparams(ns_steps=65)),
                       ([(0, 512)], malt.hparams())):
        with pytest.raises(malt.MaltError):
            malt.malt_ns_tables(shapes, hp)
    assert len(malt.malt_ns_tables([], malt.hparams())) == 0
