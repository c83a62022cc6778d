"""Every entry of profiles/counters.json is borne out by the summary that it cites, and covers the headers whose
device code its kernel takes in."""
import json
import os
import re

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def entries():
    with open(os.path.join(ROOT, "profiles", "counters.json")) as f:
        return json.load(f)


@pytest.mark.parametrize("kernel", sorted(entries()))
def test_the_summary_has_the_entrys_figures(kernel):
    e = entries()[kernel]
    with open(os.path.join(ROOT, e["summary"])) as f:
        table = "\n".join(line for line in f.read().replace(",", "").split("\n") if line.startswith("|"))
    assert re.search(r"\*\*%.0f( per |\*\*)" % e["warp_inst_per_unit"], table)
    assert "(%.0f B per " % e["dram_bytes_per_unit"] in table


@pytest.mark.parametrize("kernel", sorted(entries()))
def test_the_sources_hold_every_header_they_include(kernel):
    e = entries()[kernel]
    have = {os.path.basename(s) for s in e["sources"]}
    for src in e["sources"]:
        with open(os.path.join(ROOT, src)) as f:
            for name in re.findall(r'#include "(build_\w+\.cuh|mdp_internal\.cuh)"', f.read()):
                assert name in have, (src, name)
