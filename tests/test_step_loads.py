"""CPU: how the step kernels (csrc/lpb_step.h) read the block that the previous
kernel of an interval writes.  They are launched while that kernel runs, so the
block is not read-only for their lifetime: every gather of it goes through one
helper, which uses plain loads."""
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_the_gathered_block_is_read_by_plain_loads():
    with open(os.path.join(ROOT, "paper_2601_21990_gb300", "csrc", "lpb_step.h")) as f:
        text = re.sub(r"//[^\n]*", "", f.read())
    helper = re.search(r"void ld_iterate\([^{]*\{[^}]*\}", text)
    assert helper and "ldv(" in helper.group(0) and "ldg" not in helper.group(0)
    # no other load takes an address made from src
    rest = text.replace(helper.group(0), "")
    for load in re.findall(r"\b(?:__ld\w+|ld\w+)\s*\([^;]*;", rest):
        assert load.startswith("ld_iterate(") or not re.search(r"\bsrc\b", load), load
    assert re.search(r"\bld_iterate\(src,", rest)
