"""How the kernels of a step read memory, from the sources (no GPU). They are
launched with programmatic serialization: each is live while the one before it
still writes, and only its wait orders the two. The non-coherent path (__ldg,
ld.global.nc, a const __restrict__ kernel parameter) promises that nothing writes
the memory while the kernel lives, which holds for the tables uploaded at init
alone; and a load that is neither plain nor a volatile asm need not stay behind the
wait. A broken promise shows as a stale clip coefficient or addend, if at all, so
the sources are held to the rule themselves."""
from __future__ import annotations

import glob
import os
import re

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = sorted(glob.glob(os.path.join(ROOT, "paper_2606_30634_gb300", "csrc", "*.cu*")))
# what the two readers of init's tables may be given
TABLES = re.compile(r"^(begin|pkt_begin|a\.ch\.begin|a\.tile_begin|tiles)\b")


def code(path):
    text = re.sub(r"/\*.*?\*/", "", open(path).read(), flags=re.S)
    return re.sub(r"//[^\n]*", "", text)


def enclosing(text, pos):
    """Name of the function whose definition precedes pos most closely."""
    names = re.findall(r"__device__ __forceinline__ [\w ]+?(\w+)\(", text[:pos])
    return names[-1] if names else None


@pytest.mark.parametrize("path", CSRC, ids=[os.path.basename(p) for p in CSRC])
def test_non_coherent_loads_are_of_init_tables(path):
    text = code(path)
    for m in re.finditer(r"__ldg\(|ld\.global\.nc", text):
        assert enclosing(text, m.start()) in ("ld_table", "load_tile"), text[m.start():][:60]
    for m in re.finditer(r"(?<!I )(?<!int4 )\b(?:ld_table|load_tile)\(([^)]*)\)", text):
        assert TABLES.match(m.group(1)), m.group(0)
    for m in re.finditer(r"__global__ .*?\)\s*\{", text, flags=re.S):
        assert "__restrict__" not in m.group(0).split("{")[0], m.group(0)[:80]


@pytest.mark.parametrize("path", CSRC, ids=[os.path.basename(p) for p in CSRC])
def test_global_loads_stay_behind_the_wait(path):
    text = code(path)
    assert not re.search(r"__ld(cs|cg|ca|lu|cv)\(", text)
    for m in re.finditer(r"\"ld\.global\.", text):
        assert re.search(r"asm volatile\(\s*$", text[:m.start()]), text[m.start():][:60]


def test_the_rule_covers_every_kernel_source():
    assert {"dpo_device.cuh", "dpo_gemm.cuh", "dpo_muon.cu", "dpo_noalloc.cu"} <= {
        os.path.basename(p) for p in CSRC}
