"""The tile scan's word pair (work items, gate of the plain kernel): every
allocation of it holds the words that k_tile_scan writes."""
import os
import re

from paper_1409_5574_gb300 import build


def _read(name):
    with open(os.path.join(build.CSRC, name)) as f:
        return f.read()


def test_every_work_count_holds_the_words_the_scan_writes():
    kernel = _read("tile_sort.cu").split("k_tile_scan(", 1)[1].split("\n}\n", 1)[0]
    written = [int(k) for k in re.findall(r"\bwork_count\[(\d+)\] = ", kernel)]
    assert written and "*work_count =" not in kernel
    named = dict(re.findall(r"constexpr int (\w+) = (\d+);", _read("prad_internal.h")))
    sizes = re.findall(r"cudaMalloc\(&b\.work_count, (?:(\w+) \* )?sizeof\(unsigned int\)\)",
                       _read("prad_api.cu"))
    assert len(sizes) == 2  # (the FP64 sort's and the binning's)
    for words in sizes:
        assert int(named.get(words, words) or 1) > max(written), words
