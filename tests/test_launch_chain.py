"""What the sources owe to kernels that are launched while the one before them still runs (cowa::launch_chained)."""
import glob
import os
import re

import paper_2609_32704_b200 as cowa

CSRC = os.path.join(os.path.dirname(cowa.__file__), "csrc")


def sources():
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        with open(path) as f:
            yield os.path.basename(path), re.sub(r"//[^\n]*", "", f.read())


def test_no_load_takes_the_non_coherent_path():
    found = [(name, m) for name, text in sources() for m in re.findall(r"\.nc\b|__ldg\b|__restrict__", text)]
    assert not found


def test_every_chained_kernel_waits_for_the_one_before_it():
    kernels = 0
    for name, text in sources():
        for m in re.finditer(r"__global__[^;{]*?(cowa_\w+_kernel)\s*\([^{;]*\)\s*\{", text):
            if re.search(m.group(1) + r"(<[^;]*>)?<<<", text):
                continue  # launched the plain way: starts when everything before it is complete
            body = text[m.end():text.index("\n}\n", m.end())]
            assert re.search(r"\bgrid_(enter|wait)\(\)", body), (name, m.group(1))
            kernels += 1
    assert kernels >= 10
