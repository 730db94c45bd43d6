"""The finer splits of a mixed step's last rows keep the step at four decode
splits an SM (CPU): steps below, at and above the limit, where the plain plan
is under it and halving the whole last third would pass it."""
import pytest

from test_decode_tail_plan import _run, checker  # noqa: F401


@pytest.mark.parametrize("sms", [152, 31])
def test_at_most_four_splits_an_sm(checker, sms):  # noqa: F811
    cases = [(hq, hk, [1] * n + [512], [ctx] * n + [1512])
             for hq, hk in ((32, 8), (64, 8), (16, 2), (8, 8)) for n in (3, 16, 30, 50, 60, 70, 76, 77, 110, 130, 250)
             for ctx in (2100, 3200, 4000, 30000)]
    halved = 0
    for case, line in zip(cases, _run(checker, cases, sms)):
        assert line.startswith("ok"), (case, line)
        plain, fine = (int(x) for x in line.split()[1:])
        assert plain <= fine <= max(plain, 4 * sms), (case, line)
        halved += fine > plain
    assert halved >= 20  # (the rule is at work)
