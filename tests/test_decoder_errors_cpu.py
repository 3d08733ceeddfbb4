"""Who is told of a decoder kernel's bounded wait that ran out: the device's
error word is cleared by reading it, so what was read is kept for every reader
(host arithmetic, on a stand-in for the library's call)."""
import types

import pytest
import torch

from paper_2605_30574_gb300 import decoder as K


@pytest.fixture
def words(monkeypatch):
    """The devices' words, and the calls that read (and clear) them."""
    state = types.SimpleNamespace(word={0: 0, 1: 0}, device=0, rc=0)

    def decoder_error(ref):
        ref._obj.value, state.word[state.device] = state.word[state.device], 0
        return state.rc

    monkeypatch.setattr(K, "_LIB", types.SimpleNamespace(decoder_error=decoder_error))
    monkeypatch.setattr(K, "_records", {})
    monkeypatch.setattr(K, "_reader", K.ErrorReader(fresh=False))
    monkeypatch.setattr(torch.cuda, "current_device", lambda: state.device)
    return state


def test_every_reader_is_told_once(words):
    a, b = K.ErrorReader(), K.ErrorReader()
    a.check()
    words.word[0] = 0x10
    with pytest.raises(RuntimeError, match="0x10"):
        a.check()
    a.check()                                   # told
    words.word[0] = 0x2
    for reader in (b.check, K.check_device_error):
        with pytest.raises(RuntimeError, match="0x10, 0x2"):
            reader()
        reader()
    with pytest.raises(RuntimeError, match="word 0x2$"):
        a.check()


def test_a_new_reader_is_not_told_of_what_was_before_it(words):
    old = K.ErrorReader()
    words.word[0] = 0x4
    new = K.ErrorReader()
    new.check()
    with pytest.raises(RuntimeError, match="0x4"):
        old.check()
    with pytest.raises(RuntimeError, match="0x4"):
        K.check_device_error()


def test_devices_are_apart(words):
    r = K.ErrorReader()
    words.word[1] = 0x8
    r.check()
    words.device = 1
    with pytest.raises(RuntimeError, match="0x8"):
        r.check()


def test_a_failed_read_is_not_a_record(words):
    r = K.ErrorReader()
    words.rc = 700
    with pytest.raises(RuntimeError, match="CUDA error 700"):
        r.check()
    words.rc = 0
    r.check()
