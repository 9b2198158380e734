"""The opt-in to more than 48 KB of shared memory is an attribute of a kernel on one device.
A launcher that remembers a kernel's occupancy without the device skips the opt-in on every
device but the first, and its launches fail there.  So there is one cache of occupancies,
keyed by the device too, and the only other place that sets the attribute does so before
every launch.  (One GPU cannot show the failure, so the sources are checked.)"""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2107_05395_gb300", "csrc")


def function_around(text, pos):
    """The text from the last line that starts in column 0 and opens a function to the next
    line that closes one."""
    start = [m.start() for m in re.finditer(r"^[a-z].*\(", text, re.M) if m.start() < pos][-1]
    return text[start:text.index("\n}", pos)]


def test_one_cache_of_occupancies_keyed_by_device():
    sites = {}
    for name in sorted(os.listdir(CSRC)):
        with open(os.path.join(CSRC, name)) as fh:
            text = fh.read()
        for m in re.finditer(r"cudaFuncSetAttribute\(", text):
            sites.setdefault(name, []).append(function_around(text, m.start()))
    assert sorted((k, len(v)) for k, v in sites.items()) == [("refine.cu", 1), ("sweep.cu", 1)]
    assert sites["refine.cu"][0].startswith("int launch_one_group(")
    assert "find(" not in sites["refine.cu"][0]  # no cache
    occ = sites["sweep.cu"][0]
    assert occ.startswith("int kernel_occupancy(")
    key = re.search(r"key = std::make_tuple\((.*)\);", occ).group(1)
    assert {"kernel", "device", "threads", "smem"} <= {a.strip() for a in key.split(",")}
