"""Kernels that may start while the one before them still runs (those that call pdl_wait): what that one writes must not be read
as memory that does not change during the kernel. So no `const T* __restrict__` parameter but the tables that are written
once, and no __ldg, in these kernels and in the device functions of the files with the particle kernels."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1506_03737_gb300", "csrc")
TABLES = {"tw", "sinc2", "amp_of_n2"}
PARTICLES = {"pm_kernels.cu", "ics_kernels.cu", "noalloc.cu"}


def functions(text):
    """(qualifier, name, parameters, body) of the __global__ and __device__ function definitions."""
    for m in re.finditer(r"\b__(global|device)__\b", text):
        head = re.match(r"__(?:global|device)__(?:\s+__\w+__(?:\([^;{}]*?\)\s*(?=void|\w))?)*[^;{}()]*?(\w+)\s*\(", text[m.start():])
        if not head:
            continue
        i = m.start() + head.end()
        depth, j = 1, i
        while depth:
            depth += {"(": 1, ")": -1}.get(text[j], 0)
            j += 1
        params = text[i:j - 1]
        rest = re.match(r"\s*(const\s*)?\{", text[j:])
        if not rest:
            continue
        k = j + rest.end()
        depth, b = 1, k
        while depth:
            depth += {"{": 1, "}": -1}.get(text[b], 0)
            b += 1
        yield m.group(1), head.group(1), params, text[k:b]


def test_overlapping_kernels_read_through_plain_pointers():
    waiting, bad = set(), []
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        name = os.path.basename(path)
        text = re.sub(r"//[^\n]*", "", open(path).read())
        text = re.sub(r"__launch_bounds__\((?:[^()]|\([^()]*\))*\)", "", text)
        for kind, fn, params, body in functions(text):
            waits = kind == "global" and "pdl_wait()" in body
            if waits:
                waiting.add(fn)
            if waits or (kind == "device" and name in PARTICLES):
                bad += [f"{name}: {fn}({p})" for p in re.findall(r"const\s+[\w ]+\*\s*__restrict__\s*(\w+)", params) if p not in TABLES]
                bad += [f"{name}: {fn} __ldg" for _ in re.findall(r"__ldg\s*\(", body)]
    assert {"k_deposit", "k_gather_kick_drift", "k_conv", "k_adam", "k2_fz", "k2_fx_fwd", "k2_fy_box", "k_deposit_xyz"} <= waiting
    assert not bad, bad
