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
