"""Admission of a backlog by lanes: with a permit for each lane, every request behind a slow one
completes; with one for the whole batch, none of the next batch does.  A lane that sets a busy bit
without looking publishes over another's request."""
import pytest

from oracle import model_check as mc


@pytest.mark.parametrize("kw,nproc", [(dict(slots=2, lanes=2), 3), (dict(slots=2, lanes=1), 4),
                                      (dict(slots=1, lanes=1, requests=4, slow=-1), 4),
                                      (dict(slots=3, lanes=1, slow=2), 3), (dict(slots=4, lanes=2, slow=1), 5),
                                      (dict(slots=3, lanes=2, slow=1), 3), (dict(slots=3, lanes=3, requests=6), 4)])
def test_every_request_completes(kw, nproc):
    r = mc.check(mc.ServeAdmission(**kw), nproc, 1)
    assert r.ok, r.violation


@pytest.mark.parametrize("kw,nproc", [(dict(slots=2, lanes=2), 3), (dict(slots=3, lanes=3, requests=6), 4)])
def test_permit_for_the_batch_is_caught(kw, nproc):
    r = mc.check(mc.ServeAdmission(broken="batch_permits", **kw), nproc, 1)
    assert not r.ok and "no final state" in r.violation


@pytest.mark.parametrize("lanes,nproc", [(2, 3), (1, 4)])
def test_blind_set_is_caught(lanes, nproc):
    r = mc.check(mc.ServeAdmission(slots=2, lanes=lanes, broken="blind_set"), nproc, 1)
    assert not r.ok and "published over" in r.violation
