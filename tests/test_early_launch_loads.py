"""Kernels that may be launched before the kernel ahead of them has ended (programmatic dependent
launch) read global memory that kernel may still be writing. So they wait first, and their loads are
ordinary ones: __ldg, ld.global.nc and plain reads through a const __restrict__ pointer are defined
only for data that does not change during the kernel's life, and may be moved ahead of the wait."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2106_08034_gb300", "csrc")


def _source(path):
    src = re.sub(r"/\*.*?\*/", "", open(path).read(), flags=re.S)
    return re.sub(r"//[^\n]*", "", src)


SOURCES = {os.path.basename(p): _source(p) for p in glob.glob(os.path.join(CSRC, "*.cu*"))}


def _kernels():
    """(file, name, parameters, body) of every __global__ function."""
    for name, src in sorted(SOURCES.items()):
        for m in re.finditer(r"__global__\s+void\b", src):
            i = m.end()
            while True:  # skip __launch_bounds__(...) up to the parameter list
                k = re.compile(r"\s*(\w+)\s*\(").match(src, i)
                depth, j = 1, k.end()
                while depth:
                    depth += {"(": 1, ")": -1}.get(src[j], 0)
                    j += 1
                if k.group(1) != "__launch_bounds__":
                    break
                i = j
            params = src[k.end():j - 1]
            b = src.index("{", j)
            depth, e = 1, b + 1
            while depth:
                depth += {"{": 1, "}": -1}.get(src[e], 0)
                e += 1
            yield name, k.group(1), params, src[b:e]


KERNELS = list(_kernels())
LAUNCHED_EARLY = sorted({n for src in SOURCES.values()
                         for n in re.findall(r"launch_kernel\((?:\w+ \? \(?)*(k_\w+)", src)})


def test_the_kernels_are_found():
    names = {k[1] for k in KERNELS}
    assert set(LAUNCHED_EARLY) <= names
    assert {"k_update", "k_blend", "k_blend_tma", "k_blend_tma2", "k_blend_tma2h", "k_update_ext", "k_blend_ext",
            "k_blend_ext2", "k_read_state", "k_write_state", "k_reconstruct", "k_velocity",
            "k_render_vpt"} == set(LAUNCHED_EARLY)


@pytest.mark.parametrize("name", sorted(SOURCES))
def test_no_non_coherent_loads(name):
    assert not re.search(r"__ldg\b|ld\.global\.nc|__ldlu\b", SOURCES[name])


@pytest.mark.parametrize("kernel", LAUNCHED_EARLY)
def test_kernels_launched_early_wait_and_promise_nothing(kernel):
    (file, _, params, body), = [k for k in KERNELS if k[1] == kernel]
    assert not re.search(r"const\s+\w+\s*\*\s*__restrict__", params), file
    wait = body.index("pdl_wait()")
    for touch in ("ld_global(", "tma_load", "tma_prefetch", ".load(", ".store(", "update_any", "blend_tile"):
        first = body.find(touch)
        lam = re.search(r"auto (?:fill|stage) = \[&\]", body)  # helpers defined ahead of the wait, called behind it
        if first >= 0 and lam and first > lam.start() and first < wait:
            first = body.find(touch, body.index("};", lam.start()))
        assert first < 0 or first > wait, (kernel, touch)


@pytest.mark.parametrize("kernel", ["k_reconstruct", "k_velocity", "k_render_vpt"])
def test_input_steps_let_the_next_kernel_in_as_they_end(kernel):
    """On small images all their CTAs are resident at once; let in earlier, the next kernel's would
    crowd on the SMs that are free first."""
    (_, _, _, body), = [k for k in KERNELS if k[1] == kernel]
    assert "pdl_wait()" in body and "pdl_next" not in body


def test_work_list_kernels_are_launched_plainly_and_read_no_hint():
    """Their parameters lie in global memory: the hint of pdl_next would be a load in every tile."""
    src = SOURCES["wrls_batch.cu"]
    assert "launch_kernel(" not in src and "pdl_" not in src
    assert re.findall(r"(?:update_any|blend_tile)<([^>]*)>", src) == ["SV, true", "SV, TH, R, MODE, true"]
    assert len(re.findall(r"if constexpr \(!PERSIST\) pdl_next\(kp\);", SOURCES["wrls_tiles.cuh"])) == 3
    assert len(re.findall(r"\bpdl_next\(", SOURCES["wrls_tiles.cuh"])) == 3
