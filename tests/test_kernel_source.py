"""CPU checks of the decode kernels' source, for rules that a run cannot show to
hold: a broken one is a race that is usually won by time."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1606_00519_gb300", "csrc")


def source(name):
    with open(os.path.join(CSRC, name)) as f:
        return re.sub(r"//.*", "", f.read())


def functions(text):
    """{name: body} of the definitions that start at the left margin."""
    found = {}
    for m in re.finditer(r"^(?:static |template <[^\n]*>\n)*[^\s#}/][^;{}]*?(\w+)\([^;{}]*\)\s*\{\n(.*?)^\}", text, re.M | re.S):
        found[m.group(1)] = m.group(2)
    return found


@pytest.mark.parametrize("name", ["gmp_tile.cu", "gmp_decode.cu"])
def test_waits_cover_the_copies(name):
    # cp.async.wait_group waits for committed copies only: code that copies and
    # waits by groups also commits what it copied
    users = 0
    for fn, body in functions(source(name)).items():
        if "cp_async_wait" not in body:
            continue
        users += 1
        copies = [m.start() for m in re.finditer(r"\bcp_async16(?:_if)?\(", body)]
        commits = [m.start() for m in re.finditer(r"\bcp_async_commit\(", body)]
        assert copies and commits and commits[-1] > copies[-1], fn
    assert users >= 1


def test_one_warp_reads_what_a_caller_can_change():
    # warps that share a block's barriers take the block's header, descriptor
    # and index entry from the one warp that read them, and the choice between
    # two launches is read from a device word, not worked out by each CTA
    text = source("gmp_tile.cu")
    text = re.sub(r"__launch_bounds__\([^)]*\)+ ", "", text)
    found = functions(text)
    kernels = {k: v for k, v in found.items() if k in ("coop_kernel", "tile_kernel")}
    assert len(kernels) == 2 and [k for k, v in found.items() if "open_block(" in v] == ["take_block"]
    for body in kernels.values():
        assert not re.search(r"gmp_file_desc|find_file|wait_input|ld_u32_nc|->comp|\.comp\b", body)
        assert len(re.findall(r"\btake_block<", body)) == 1
        guard = body[:body.index("take_block<")]
        assert re.search(r"if \((half == 0|t < 32)\) \{(?:[^{}]|\{[^{}]*\})*$", guard)
    assert "takes_coop" not in text and "route_of" not in text


def test_sizes_read_twice_are_bounded():
    # the sub-block table is read once, where its totals are checked; records
    # written one by one are read a second time, and cut to what is left
    found = functions(source("gmp_tile.cu"))
    assert [k for k, v in found.items() if re.search(r"192u? \+ 12u? \* j", v)] == ["sub_block_table"]
    assert len(re.findall(r"192u? \+ 12u? \* j", source("gmp_decode.cu"))) == 1
    body = found["slow_group"]
    assert "out_bytes - w.g0" in body and "lits_end - lits" in body and "dist <= w.g0" in body
