"""Argument forms of the C module of the per-step calls (no GPU needed): what
it takes in place, and what it leaves to the ctypes path."""
import numpy as np
import pytest

import paper_2607_10582_gb300 as md
from paper_2607_10582_gb300 import build as mdbuild


@pytest.fixture(scope="module")
def calls():
    mdbuild.build()
    return md._binding()


def per_step_calls(calls, regs, batch=2):
    """The status of each call that takes labels, on a null handle: an error
    when the labels are taken in place, None when they are not."""
    return [calls.decode_step(None, batch, None, None, None, regs, None),
            calls.decode_layer(None, 0, batch, None, None, None, regs, None)]


@pytest.mark.parametrize("regs", [np.array([5, 6], np.uint8), bytearray([5, 6]), memoryview(bytes([5, 6]))])
def test_labels_taken_in_place(calls, regs):
    assert per_step_calls(calls, regs) == [md.MD_ERR_INVALID_ARG] * 2


@pytest.mark.parametrize("regs", [b"56", b"\x05\x06", [5, 6], np.array([5, 6]), np.array([5, 6], np.int8),
                                  np.array([5, 0, 6, 0], np.uint8)[::2], np.array([[5, 6]], np.uint8), np.uint8(5)])
def test_labels_left_to_the_ctypes_path(calls, regs):
    """Byte strings among them: numpy reads those as text, so "6" is region 6
    there and anything that is no number is refused."""
    assert per_step_calls(calls, regs) == [None, None]


def test_labels_fewer_than_the_batch_are_not_taken(calls):
    """The library reads one label per sequence: a shorter array is left to the
    caller's check, except by the layers after the first, which read none."""
    short = np.array([6], np.uint8)
    assert per_step_calls(calls, short) == [None, None]
    assert calls.decode_layer(None, 1, 2, None, None, None, short, None) == md.MD_ERR_INVALID_ARG
    assert per_step_calls(calls, short, batch=-1) == [md.MD_ERR_INVALID_ARG] * 2
    torch = pytest.importorskip("torch")
    x = torch.zeros(4)
    assert calls.decode_step_host(None, 2, x, x, x, short, x) is None
    assert calls.decode_step_host(None, 1, x, x, x, short, x) == md.MD_ERR_INVALID_ARG


@pytest.mark.parametrize("regs", [[6], np.array([6], np.uint8), []])
def test_labels_fewer_than_the_batch_are_refused(calls, regs):
    """By either path, before the library reads past the array's end; a batch
    that the handle refuses anyway is left to it."""
    torch = pytest.importorskip("torch")
    c = object.__new__(md.Cache)
    c.h = c._hv = None
    c._b, c.max_batch = calls, 4
    x = torch.zeros(4)
    for call in (lambda b: c.decode_step(b, None, None, None, regs, None),
                 lambda b: c.decode_layer(0, b, None, None, None, regs, None),
                 lambda b: c.decode_step_host(b, x, x, x, regs, x)):
        with pytest.raises(md.MemDecayError, match="labels") as e:
            call(2)
        assert e.value.status == md.MD_ERR_INVALID_ARG
        with pytest.raises(md.MemDecayError, match="null handle") as e:
            call(5)
        assert e.value.status == md.MD_ERR_INVALID_ARG
    with pytest.raises(md.MemDecayError, match="null handle"):      # layers after the first read no labels
        c.decode_layer(1, 2, None, None, None, regs, None)


def test_fewer_insertion_steps_than_labels_are_refused():
    """The library reads one insertion step per label."""
    c = object.__new__(md.Cache)
    c.h = None
    for steps in ([0], np.zeros(1, np.int32), []):
        with pytest.raises(md.MemDecayError, match="insertion steps") as e:
            c.append_tokens(0, [5, 6], None, None, steps)
        assert e.value.status == md.MD_ERR_INVALID_ARG
    with pytest.raises(md.MemDecayError, match="null handle"):
        c.append_tokens(0, [5, 6], None, None, [0, 0])
