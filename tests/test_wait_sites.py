"""Every bounded wait on the device has a code of its own, and the codes of a kernel share their leading digit with no other kernel's:
what `ago_subgraph_status` reports after a wait that ran out names kernel and place. Read from the sources."""
import collections
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2212_01005_b200", "csrc")


def test_wait_codes_name_one_place_each():
    sites = collections.defaultdict(list)
    for path in glob.glob(os.path.join(CSRC, "*.cu")):
        text = re.sub(r"//[^\n]*", "", open(path).read())
        waits = re.findall(r"\bmbar_wait(?:_poll)?\([^;]*?status, (\w+)\)", text)
        assert len(waits) == len(re.findall(r"\bmbar_wait(?:_poll)?\(", text)), path
        for code in waits:
            assert re.fullmatch(r"0x[0-9a-f]{3}", code), (path, code)
            sites[code].append(os.path.basename(path))
    assert len(sites) > 50
    assert not {c: f for c, f in sites.items() if len(f) > 1}
    kernels = collections.defaultdict(set)
    for code, files in sites.items():
        kernels[code[:3]].update(files)
    assert all(len(f) == 1 for f in kernels.values()), dict(kernels)
