"""Kernels that may start while their predecessor runs (programmatic dependent launch) read what it wrote only behind their wait and only by
ordinary loads: the read-only path is for data that nobody writes while the kernel is resident.  Checked on the sources, since no run shows
a load that happened to come late enough."""
import os
import re

import pytest

from paper_2511_11248_b200 import build

WAIT = 'asm volatile("griddepcontrol.wait;"'
# weights, which no kernel that may still be running writes (include/tman.h, stream order of the packed buffer)
WEIGHTS = re.compile(r"__ldg\((p\.packed|p\.scales|p\.zeros|psc|pz|reinterpret_cast<const uint(4|32_t) \*>\(p\.packed)")


def kernels_with_a_wait():
    found = []
    for name in sorted(os.listdir(build.CSRC)):
        if not name.endswith((".cu", ".cuh")):
            continue
        with open(os.path.join(build.CSRC, name)) as f:
            text = re.sub(r"//[^\n]*", "", f.read())
        for m in re.finditer(r"__global__ void[^;{]*?(\w+)\s*\((?P<args>[^)]*)\)\s*\{(?P<body>.*?)\n\}", text, re.S):
            if WAIT in m["body"]:
                found.append((name, m[1], m["args"], m["body"]))
    return found


def test_every_kernel_with_a_wait_is_found():
    assert {k[1] for k in kernels_with_a_wait()} == {"mpgemv_kernel", "decode_mma_kernel", "decode_digits_kernel", "mpgemm_kernel", "quantize_rows_regs_kernel"}


@pytest.mark.parametrize("name,kernel,args,body", kernels_with_a_wait(), ids=lambda v: v if isinstance(v, str) and v.endswith("_kernel") else "")
def test_nothing_a_predecessor_wrote_is_read_by_the_read_only_path(name, kernel, args, body):
    after = body[body.index(WAIT):]
    loads = [after[m.start():after.index(";", m.start())] for m in re.finditer(r"__ldg\(|ld\.global\.nc|__ldlu\(", after)]
    assert [v for v in loads if not WEIGHTS.match(v)] == []
    assert not re.search(r"const [^,]*__restrict__", args)          # (the compiler may read through it by the read-only path on its own)
    assert "row_scale" not in body[:body.index(WAIT)]
