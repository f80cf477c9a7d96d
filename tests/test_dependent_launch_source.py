"""Kernels that may run beside their predecessor (programmatic dependent launch, pdl.cuh)
read what it writes through plain pointers: loads through a __restrict__ parameter may be
moved above the wait, and a `const __restrict__` one or __ldg reads non-coherently."""
import os
import re

from paper_2107_11311_gb300 import build

CONSTANT = {"pnet", "sinfo", "types"}  # written by no kernel of an evaluation
# written or atomically updated by the kernel, and read by it at most after it wrote them
OUTPUTS = {"k_scan_cells": {"start"}, "k_scatter": {"pos4", "perm"},
           "k_list_build": {"rows", "codes", "count", "F4", "stats", "err"},
           "k_potential_list": {"F4", "eatom", "G_out", "e_part", "vir_part", "vir_atom", "stats", "err", "work"},
           "k_finalize": {"result"}, "k_md_kick_finish": {"vl_flag", "vl_builds"},
           "k_md_turn": {"tmp4", "cell_of", "cell_start", "stats", "err"}}


def _kernels():
    for f in sorted(os.listdir(build.CSRC)):
        if not f.endswith((".cu", ".cuh")) or f == "pdl.cuh":
            continue
        src = re.sub(r"//[^\n]*", "", open(os.path.join(build.CSRC, f)).read())
        for m in re.finditer(r"__global__\s+void\s+(?:__launch_bounds__\([^{;]*?\)\s+)?(\w+)\s*\(", src):
            depth, i = 1, m.end()
            while depth:
                depth += {"(": 1, ")": -1}.get(src[i], 0)
                i += 1
            if not src[i:].lstrip().startswith("{"):
                continue  # a declaration
            params, depth, j = src[m.end():i - 1], 0, src.index("{", i)
            k = j
            while True:
                depth += {"{": 1, "}": -1}.get(src[k], 0)
                k += 1
                if depth == 0:
                    break
            yield m.group(1), params, src[j:k]


def test_dependent_kernels_read_through_plain_pointers():
    launched = set()
    for f in os.listdir(build.CSRC):
        if f.endswith((".cu", ".cuh")):
            src = open(os.path.join(build.CSRC, f)).read()
            launched |= set(re.findall(r"launch_after\(\s*[^,]+,\s*(k_\w+)", src))
    seen = set()
    for name, params, body in _kernels():
        if "pdl_wait()" not in body:
            assert name not in launched, f"{name} is launched early and does not wait"
            continue
        seen.add(name)
        assert "__ldg(" not in body, name
        for p in (re.sub(r"\s+", " ", q).strip() for q in params.split(",")):
            q = re.match(r"(const )?.*\*\s*__restrict__ (\w+)$", p)
            if q and q.group(2) not in CONSTANT:  # outputs only: never read (by a plain load) in the kernel
                assert not q.group(1), f"{name}: {p}"
                assert q.group(2) in OUTPUTS.get(name, ()), f"{name}: {p}"
    assert launched <= seen and {"k_list_build", "k_potential_list", "k_scatter", "k_finalize"} <= seen
