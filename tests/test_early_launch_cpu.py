"""Kernels that are launched while the kernel before them still runs read their tensors by plain loads.  The read-only path (``__ldg``,
``ld.global.nc``, and what the compiler makes of a ``const __restrict__`` pointer) is for memory that nothing writes during the
kernel's lifetime, and there the kernel before may still be writing it.  A plan's constants may be read that way."""
import os
import re

import pytest

from paper_2006_11735_b200.build import CSRC

SOURCES = {f: open(os.path.join(CSRC, f)).read() for f in sorted(os.listdir(CSRC)) if f.endswith((".cu", ".cuh"))}
# files all of whose kernels come up early (launched with that attribute by umma_launch and the picture kernel's launch)
EARLY_FILES = [f for f in SOURCES if f.startswith("umma_")] + ["kernel_picture.cu", "kernel_pool.cu"]
CONSTANT = re.compile(r"(cap|ua?\.c_\w+|u\.w|a\.(w|bias|mul|shift|h_i)|layers\.l\[l\]\.c_a)\b")


def _kernels(text):
    """name -> (parameters, body) of the kernels that a file defines."""
    out = {}
    for m in re.finditer(r"__global__[^;{]*?\b(\w+_kernel)\(", text):
        i, depth = m.end(), 1
        while depth:                                             # the parameters' end
            depth += {"(": 1, ")": -1}.get(text[i], 0)
            i += 1
        if not text[i:].lstrip().startswith("{"):
            continue                                             # a declaration
        start = j = text.index("{", i)
        depth = 0
        while True:
            depth += {"{": 1, "}": -1}.get(text[j], 0)
            j += 1
            if not depth:
                break
        out[m.group(1)] = (text[m.end():i], text[start:j])
    return out


EARLY = sorted({name for text in SOURCES.values() for m in re.finditer(r"launch_kernel\(((?:[^,;]|<[^>]*>)*?), true,", text)
                for name in re.findall(r"\w+_kernel", m.group(1))} - {"collect_kernel", "settle_kernel"})
# (collect_kernel's tensor is complete before the kernel in front of it, which it overlaps, has started; settle_kernel reads past the caches that
# are not coherent)


def _constants_only(text, where):
    assert not re.search(r"\.nc\b", text), where
    for m in re.finditer(r"__ldg\((\((?:const )?\w+ \*\))?\(?", text):
        assert CONSTANT.match(text, m.end()), (where, text[m.start():m.start() + 80])


def test_the_kernels_are_found():
    assert {"stem_repack_kernel", "stem_repack_wide_kernel", "rows_repack_kernel", "stem_pool_kernel", "add_requant_fast_kernel", "maxpool_3x3s2_kernel",
            "maxpool_3x3s2_wide_kernel", "avgpool16_kernel", "few_kernel"} == set(EARLY)


@pytest.mark.parametrize("name", EARLY)
def test_a_kernel_that_comes_up_early_reads_its_tensors_by_plain_loads(name):
    (params, body), = [k[name] for k in map(_kernels, SOURCES.values()) if name in k]
    assert "__restrict__" not in params
    assert "grid_dep_wait()" in body
    _constants_only(body, name)


@pytest.mark.parametrize("file", EARLY_FILES)
def test_the_tensor_core_kernels_read_their_tensors_by_plain_loads(file):
    assert "__restrict__" not in SOURCES[file]
    _constants_only(SOURCES[file], file)
