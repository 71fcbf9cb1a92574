"""Serving: what the claims may do to a slot while the host installs a code."""
import pytest

from paper_2603_29942_gb300 import _binding as B

TRANSIT = 1 << 39  # the counter's task index while the host writes a code into a slot


@pytest.mark.parametrize("gen", [0, 1, 0xFFFF])
def test_a_code_being_installed_is_not_marked_used_up(gen):
    """A claim that meets the transition value (or comes after other claims on
    it) finds no task, as past the end of a schedule; only there may it mark
    the code used up, or a code that has not begun would never be searched."""
    word = gen << 48
    for claims in (0, 1, 608, 10 ** 6):
        assert B.lib().fpcode_test_marks_used_up(word | (TRANSIT + claims)) == 0
    for index in (1, 25, 2 ** 32 - 1, 2 ** 32, 2 ** 32 + 608, TRANSIT - 1):
        assert B.lib().fpcode_test_marks_used_up(word | index) == 1
