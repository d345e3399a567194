"""Flags of the CG launches, by reading the source: a launch may set the flags
that end a solve while its own blocks still run only where no other block of
it looks at them, because a block whose warps disagree about an early return
would meet its barriers with warps missing."""

import pathlib
import re

CSRC = pathlib.Path(__file__).resolve().parent.parent / "paper_0910_2950_gb300" / "csrc"


def body(source, name):
    """Text between the braces of the function `name`."""
    at = source.index("{", re.search(r"\b%s\s*\(" % name, source).end())
    depth = 0
    for i in range(at, len(source)):
        depth += {"{": 1, "}": -1}.get(source[i], 0)
        if depth == 0:
            return re.sub(r"//.*", "", source[at:i])
    raise AssertionError(name)


def test_blocks_beside_the_publishing_one_read_nothing_that_it_writes():
    source = (CSRC / "fermion.cu").read_text()
    written = set()
    for name in ("publish", "publish_iteration"):
        written |= set(re.findall(r"cgd->(\w+)(?:\[[^\]]*\])?\s*=[^=]", body(source, name)))
    assert "done" in written
    read = set(re.findall(r"cgd->(\w+)", body(source, "cg_hop_split_kernel")))
    assert read and not read & written


def test_the_flag_they_read_is_set_back_with_done():
    source = (CSRC / "fermion.cu").read_text()
    assert re.findall(r"cgd->done\s*=[^=]", source.replace(body(source, "set_done"), "")) == ["cgd->done = "]
    assert "cgd->done = 1;" in body(source, "publish")
