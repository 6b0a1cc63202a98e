"""Rules of the kernels that cannot be observed in a result: read from the sources."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2608_17442_b200", "csrc")
FILES = sorted(glob.glob(os.path.join(CSRC, "*.cu")))


def functions(text, head):
    """(name, parameters, body) of the functions whose declaration starts with `head`."""
    text = re.sub(r"//[^\n]*", "", text)
    for m in re.finditer(head, text):
        start = text.index("{", text.index("(", _name_end(text, m.end())))
        name = re.search(r"(\w+)\s*$", text[m.end():_name_end(text, m.end())]).group(1)
        depth, end = 0, start
        while True:
            depth += {"{": 1, "}": -1}.get(text[end], 0)
            end += 1
            if depth == 0:
                break
        yield name, text[_name_end(text, m.end()):start], text[start:end]


def _name_end(text, at):
    """Position of the parenthesis that opens the parameters: the attributes before the name have their own."""
    while True:
        at = text.index("(", at)
        if not re.search(r"(__launch_bounds__|__align__)\s*$", text[:at]):
            return at
        depth = 0
        while True:
            depth += {"(": 1, ")": -1}.get(text[at], 0)
            at += 1
            if depth == 0:
                break


def test_the_reader_finds_the_kernels():
    names = [n for f in FILES for n, _, _ in functions(open(f).read(), r"__global__ void")]
    assert len(names) > 45 and {"k_rows_inner", "k_small_switch", "ntt16_rows_fwd", "k_inner", "k_ct_pt_mac"} <= set(names)


@pytest.mark.parametrize("path", FILES, ids=os.path.basename)
def test_kernels_that_start_early_read_no_written_buffer_through_the_read_only_path(path):
    """A kernel that is set up while its predecessor runs waits before it touches what kernels write; a __restrict__ parameter that it only
    reads would be read through the read-only path, ahead of that wait if the compiler likes.  Words and bytes are what kernels write; the
    tables of a context (constants, twiddles, conversion matrices) have types of their own."""
    for name, params, body in functions(open(path).read(), r"__global__ void"):
        if not re.search(r"pdl_begin\(\)|SMALL_BEGIN\(|griddepcontrol\.wait", body):
            continue
        bad = [p.strip() for p in params.split(",") if "__restrict__" in p and re.search(r"\b(u64|uint64_t|uint8_t)\b", p)]
        assert not bad, (name, bad)


def test_words_that_were_read_are_handed_to_bulk_copies_in_order():
    """k_rows_inner and k_inner_tma refill shared memory that other threads have read: the copies belong to the asynchronous proxy, and the
    one who starts them learns that the others are done from a count that releases and acquires (or from a CTA barrier)."""
    seen = 0
    for f in ("inner16.cu", "ops.cu"):
        for name, _, body in functions(open(os.path.join(CSRC, f)).read(), r"__global__ void"):
            if "bulk_g2s(" in body:
                seen += 1
                assert "before_refill()" in body and not re.search(r"\batomic(Inc|Add)\(", body), name
    assert seen == 2
    common = open(os.path.join(CSRC, "common.cuh")).read()
    assert "atom.acq_rel.cta.shared::cta.inc.u32" in common and "fence.proxy.async.shared::cta" in common
