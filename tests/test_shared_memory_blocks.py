"""The grid-wide resident form's barrier block (a struct) and the shared memory
that its launch asks for come from one size (checked in the source: a launch
whose block lies past its allocation is not run)."""

import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_barrier_block_lies_inside_the_allocation():
    src = open(os.path.join(ROOT, "paper_2312_05837_gb300", "csrc", "ds_tc.cu")).read()
    body = re.search(r"struct ResBars \{(.*?)\};", src, re.S).group(1)
    slots = int(re.search(r"constexpr int kResSlots = (\d+);", src).group(1))
    size = 0
    for kind, names in re.findall(r"(uint64_t|uint32_t|int) ([^;]+);", body):
        for f in names.split(","):
            n = re.search(r"\[(\w+)\]", f)
            size += (8 if kind == "uint64_t" else 4) * (1 if n is None else slots if n[1] == "kResSlots"
                                                        else int(n[1]))
    assert size == 4 * 8 * slots + 10 * 8 + 8
    tail = re.search(r"kResTail = \(sizeof\(ResBars\) \+ 127\) / 128 \* 128", src)
    assert tail and re.search(r"int64_t region = .*kResTail\) / 1024 \* 1024;", src)
    assert re.search(r"bytes = \(size_t\)region \+ kResTail \+ 1024;", src)
    # whatever the shared memory of the device, block and slack fit beside the region
    block = (size + 127) // 128 * 128
    for optin in range(100 * 1024, 228 * 1024, 64):
        region = (optin - 1024 - block) // 1024 * 1024
        for pad in range(0, 1024, 16):  # the dynamic base's distance to a 1024-byte boundary
            assert pad + region + size <= region + block + 1024 <= optin
