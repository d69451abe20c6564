"""The order in which the tensor-core quantiser's CTAs go through an activation tensor, checked without a GPU."""
import pytest

from paper_2603_16590_b200 import binding as B

# strips of 128 channels, row tiles of 128 tokens, SMs, units left to the CTAs that do not walk in step (None: nobody does)
WALKS = [(1, 300, 148, 0),      # one strip: every CTA walks it
         (5, 24, 148, 0),       # single strips, every unit a CTA of its own
         (5, 121, 148, 0),      # walked in step; three CTAs have nothing to do
         (41, 20, 148, 82),     # single strips, three CTAs a strip; 25 CTAs take the last two rows
         (6, 70, 148, 0),       # pairs of strips
         (26, 50, 148, 130),    # pairs, the last five rows to eight CTAs
         (64, 38, 148, 256),    # groups of four, the last four rows to 20 CTAs
         (145, 3, 148, 0),      # as many strips as CTAs but three
         (200, 3, 148, None),   # more groups of strips than of CTAs: ranges
         (150, 3, 148, None), (149, 3, 148, None),
         (7, 11, 2, None), (3, 9, 1, None), (1, 1, 148, 0), (12, 40, 132, 0), (10, 1000, 132, 120)]


@pytest.mark.parametrize("strips,rows,sms,left", WALKS)
def test_units_are_taken_once_and_evenly(strips, rows, sms, left):
    walk = B.batq_debug_quantize_walk(strips, rows, sms)
    ctas = min(sms, strips * rows)
    assert len(walk) == ctas
    units = [u for w in walk for u in w]
    assert len(units) == len(set(units)) == strips * rows
    assert set(units) == {(s, r) for s in range(strips) for r in range(rows)}
    group = next(g for g in (4, 2, 1) if strips % g == 0 and ctas % g == 0)
    assert max(map(len, walk)) == -(-(strips // group * rows) // (ctas // group))   # nobody above an even share
    # in step: CTA c starts on strip c % strips (of its group) and goes down it by the CTAs of that strip
    per = ctas // group // (strips // group)
    walkers = per * strips
    assert (left is None) == (per == 0)
    if per:
        assert sum(map(len, walk[walkers:])) == left
        for w in walk[:walkers]:
            assert len({s for s, _ in w}) <= 1 and all(b[1] - a[1] == per for a, b in zip(w, w[1:]))
    # neighbouring CTAs of a group have neighbouring strips and the same rows
    for c in range(0, ctas - group + 1, group):
        for i in range(1, group):
            assert [(s + i, r) for s, r in walk[c]] == walk[c + i]


def test_every_small_shape():
    for strips in range(1, 24):
        for rows in range(1, 24):
            for sms in (1, 2, 3, 4, 6, 8, 13, 16):
                walk = B.batq_debug_quantize_walk(strips, rows, sms)
                units = [u for w in walk for u in w]
                assert len(units) == strips * rows and len(set(units)) == len(units)


def test_arguments_out_of_range():
    for args in ((0, 1, 1), (1, 0, 1), (1, 1, 0)):
        with pytest.raises(ValueError):
            B.batq_debug_quantize_walk(*args)
