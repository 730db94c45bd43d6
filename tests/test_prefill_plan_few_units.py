"""Plans of steps with few (query tile, head slot) units: every unit is cut in
equal pieces, one to a CTA, when that shortens the longest CTA.  The checker
of test_prefill_plan.py verifies every index; here also the longest CTA load
(KV tiles + 3 an item) against the equal split's."""
import pytest

from test_prefill_plan import _run, checker  # noqa: F401

ITEM = 3


# (q-heads, kv-heads, q_lens, ctx_lens, longest piece in KV tiles)
@pytest.mark.parametrize("hq,hk,q,c,most", [
    (16, 2, [512], [2048], 5),            # 32 units of 13-16 tiles
    (16, 2, [1, 1, 512], [2048, 2048, 2048], 5),  # the same beside decode splits
    (16, 2, [128], [2048], 4),            # 8 units of 16 tiles: pieces of the minimum length
    (8, 8, [100], [700], 6),              # group 1; units of 6 tiles cut at most once
    (16, 2, [2], [128], 1),               # one tile: nothing to cut
    (32, 8, [130], [130 + 8192], 15),     # 32 units of 65-66 tiles: the cut from the front stays (4 equal pieces: 17)
])
def test_equal_pieces(checker, hq, hk, q, c, most):  # noqa: F811
    (split, whole), = _run(checker, [(hq, hk, q, c)])
    assert split.startswith("ok"), split
    assert whole.startswith("ok"), whole
    assert float(split.split()[5]) <= most + ITEM, split


@pytest.mark.parametrize("sms", [1, 2, 31, 152, 256])
def test_every_unit_count_around_the_cta_count(checker, sms):  # noqa: F811
    # units of every length around the minimum piece, as many as the CTAs and around that
    cases = [(16, 2, [128 * t], [128 * n]) for t in (1, 2, 4) for n in range(t, 14)]
    cases += [(hk, hk, [2] * k, [120 + 128 * k] * k) for hk in (1, 4) for k in (1, 7, 31, 38, 39)]
    for case, (split, whole) in zip(cases, _run(checker, cases, sms)):
        assert split.startswith("ok"), (case, split)
        assert whole.startswith("ok"), (case, whole)
