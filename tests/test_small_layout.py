"""Where the rows of the small rings lie in shared memory, with the macro as the source has it: every point has a place of its own, and in
every round the sixteen threads of a half-warp reach sixteen different banks of eight bytes."""
import os
import re

import pytest

SOURCE = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2608_17442_b200", "csrc", "small.cu")


def place(e):
    text = re.search(r"#define SM_AT\(e\) (.*)", open(SOURCE).read()).group(1)
    return eval(text, {"e": e})      # shifts, masks and exclusive or: the same operators in both languages


@pytest.mark.parametrize("log_n", [10, 11, 12])
def test_rounds_reach_sixteen_banks(log_n):
    n = 1 << log_n
    at = [place(e) for e in range(n)]
    assert sorted(at) == list(range(n))
    for stride in (n // 8, n // 64, n // 512, 1):
        for k in range(8):
            for half in range(0, n // 8, 16):
                points = [t // stride * 8 * stride + k * stride + t % stride for t in range(half, half + 16)]
                assert len({at[e] % 16 for e in points}) == 16, (stride, k, half)
            for t in range(n // 8):          # the thread's and the register's parts of a point are combined as at8 does it
                own, reg = t // stride * 8 * stride + t % stride, k * stride
                assert at[own + reg] == (at[own] ^ (at[reg] & 15)) + (at[reg] & ~15)
