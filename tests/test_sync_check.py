"""SFFN_SYNC_CHECK=1: every call looks at the environment as it is then."""
import os
import types

import pytest
import torch


@pytest.fixture
def checked():
    """Whether a call (of a library that only says yes) was followed by the check."""
    from paper_2609_31975_b200.binding import SparseFFN

    def call():
        seen = []
        x = torch.zeros(64)
        me = types.SimpleNamespace(_h=None, _gate=lambda gate: None, _stream=lambda stream: 0, _sync_check=lambda *a: seen.append(a))
        SparseFFN._call(me, lambda *a: 0, "a call", x, {}, None, x, x, "relu", x, None)
        return bool(seen)

    return call


def test_the_variable_is_heard_when_it_changes(checked, monkeypatch):
    monkeypatch.delenv("SFFN_SYNC_CHECK", raising=False)
    assert not checked()
    for value, want in (("1", True), ("0", False), ("1", True)):
        monkeypatch.setenv("SFFN_SYNC_CHECK", value)
        assert checked() == want
    monkeypatch.delenv("SFFN_SYNC_CHECK")
    assert not checked()


def test_another_environment_in_its_place_is_heard(checked, monkeypatch):
    monkeypatch.delenv("SFFN_SYNC_CHECK", raising=False)
    monkeypatch.setattr(os, "environ", {"SFFN_SYNC_CHECK": "1"})
    assert checked()
    monkeypatch.setattr(os, "environ", {})
    assert not checked()
