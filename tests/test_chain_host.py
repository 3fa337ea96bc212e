"""Kernels launched while their predecessor drains (launch_chained in
csrc/lf_internal.cuh), read as source: loads through a const __restrict__
kernel parameter may be taken for reads of memory that nobody writes during the
kernel's life and be moved ahead of chain_wait(), so no such kernel declares one
for memory that its predecessor writes."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(__file__), "..", "paper_1102_3094_gb300", "csrc")
# work lists of the ensemble: written by the host when the batch is built
HOST_TABLES = re.compile(r"const (EnsRun|EnsItem|EnsT|EnsTItem)\s*\* __restrict__")


def source(path):
    text = open(path).read()
    text = re.sub(r"/\*.*?\*/", "", text, flags=re.S)
    return re.sub(r"//[^\n]*", "", text)


def matching(text, i):
    """Index past the bracket that closes the one at text[i]."""
    pair = {"(": ")", "{": "}"}[text[i]]
    depth = 0
    for j in range(i, len(text)):
        depth += (text[j] == text[i]) - (text[j] == pair)
        if depth == 0:
            return j + 1
    raise AssertionError("unbalanced")


def files():
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")) + glob.glob(os.path.join(CSRC, "*.cuh")))


def kernels(text):
    """(name, parameters, body) of every kernel defined in `text`."""
    for m in re.finditer(r"__global__", text):
        head = re.compile(r"\b(k_\w+)\s*\(").search(text, m.end())
        if not head:
            continue
        end = matching(text, head.end() - 1)
        rest = re.match(r"\s*\{", text[end:])
        if rest:
            body = end + rest.end() - 1
            yield head.group(1), text[head.end():end - 1], text[body:matching(text, body)]


def chained():
    out = []
    for path in files():
        out += [(os.path.basename(path), *k) for k in kernels(source(path)) if "chain_wait()" in k[2]]
    return out                                   # (file, name, parameters, body)


def test_the_scan_finds_the_kernels():
    names = {k[1] for k in chained()}
    assert {"k_march2d_x2", "k_tsub2d_rows", "k_step2d_f64", "k_force3d_x2", "k_lb3d", "k_phi3d_q", "k_tsub3d_q",
            "k_ens_march2d", "k_ens_tsub2d", "k_conv3x3"} <= names


@pytest.mark.parametrize("kernel", chained(), ids=lambda k: k[1])
def test_no_restrict_parameter_for_memory_of_the_predecessor(kernel):
    assert "__restrict__" not in HOST_TABLES.sub("", kernel[2])


@pytest.mark.parametrize("path", files(), ids=os.path.basename)
def test_no_restrict_outside_kernel_parameters(path):
    """Nor on a pointer made inside a kernel or a function that kernels share."""
    text = source(path)
    for _, params, _ in kernels(text):
        text = text.replace(params, "")
    assert "__restrict__" not in text


@pytest.mark.parametrize("path", files(), ids=os.path.basename)
def test_no_launch_status_is_dropped(path):
    """A launch that is refused (its configuration or attributes) only says so in what launch_chained returns; under
    capture a graph would go without that kernel."""
    text = source(path)
    assert not re.search(r"[;{})]\s*launch_chained\(", text)
