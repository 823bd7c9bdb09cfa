"""The reuse of the serving ring's entries: the producer waits for the completed prefix.  The model
with that rule is live for every order of completion; by the number of completed requests it loses
one whose lane is slow (with one lane, completions are in order and both rules are the same)."""
import pytest

from oracle import model_check as mc


@pytest.mark.parametrize("entries,requests,lanes", [(1, 3, 2), (2, 5, 1), (2, 5, 3), (4, 6, 2)])
def test_prefix_rule_is_live(entries, requests, lanes):
    r = mc.check(mc.RingReuse(entries=entries, requests=requests), 1 + lanes, 1)
    assert r.ok, r.violation


@pytest.mark.parametrize("entries,lanes", [(2, 2), (2, 3), (4, 4)])
def test_count_rule_loses_a_request(entries, lanes):
    r = mc.check(mc.RingReuse(entries=entries, requests=entries + 2, broken="completed_count"), 1 + lanes, 1)
    assert not r.ok and "cannot reach completion" in r.violation
    assert mc.check(mc.RingReuse(entries=entries, requests=entries + 2, broken="completed_count"), 2, 1).ok
