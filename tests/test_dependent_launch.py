"""Kernels that are launched while the kernel before them still runs (launch_pdl), read in
the sources: each waits for it (pdl_wait) before its work, and declares none of its pointers
__restrict__, reads nothing through the read-only path: what they point to may still be
written when the kernel starts."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1003_0844_gb300", "csrc")


def _sources():
    out = {}
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu")) + glob.glob(os.path.join(CSRC, "*.cuh"))):
        text = open(path).read()
        out[os.path.basename(path)] = re.sub(r"//[^\n]*|/\*.*?\*/", "", text, flags=re.S)
    return out


def _closing(text, start, pair):
    depth = 0
    for i in range(start, len(text)):
        depth += (text[i] == pair[0]) - (text[i] == pair[1])
        if depth == 0:
            return i
    raise AssertionError("unbalanced " + pair)


def _kernels():
    """name -> (parameters, body) of every __global__ function."""
    found = {}
    for name, text in _sources().items():
        for m in re.finditer(r"__global__\s+void\s+(?:__launch_bounds__\((?:[^()]|\([^()]*\))*\)\s+)?(k_\w+)\s*\(", text):
            end = _closing(text, m.end() - 1, "()")
            body = text.index("{", end)
            if text[end + 1:body].strip():
                continue  # a declaration
            found[m.group(1)] = (text[m.end():end], text[body:_closing(text, body, "{}") + 1], name)
    return found


KERNELS = _kernels()


def _by_pointer():
    """Kernels that a launch names without <<<>>>: those handed to launch_pdl or a wrapper of it
    (k_pass1 and k_pass2 are launched the ordinary way through a variable)."""
    names = set()
    for text in _sources().values():
        for m in re.finditer(r"\b(k_\w+)(\s*<[\w\s,:*+]*>)?(?=\s*[,;):?])", text):
            ordinary = re.match(r"[^{}]*;[^{}]*?\bkern\s*<<<", text[m.end():]) and "launch_pdl(kern" not in re.match(
                r"[^{}]*", text[m.end():]).group(0)
            if m.group(1) in KERNELS and not ordinary:
                names.add(m.group(1))
    return names


DEPENDENT = sorted(_by_pointer() | {k for k, (_, body, _) in KERNELS.items() if "pdl_wait()" in body})


def test_the_kernels_are_found():
    assert len(KERNELS) > 40
    for name in ("k_moments", "k_passes", "k_demod_nodes", "k_stockham64_r16", "k_conv_rows", "k_fft64_cols",
                 "k_spline", "k_points_final", "k_resampled", "k_interbin_edges", "k_data32"):
        assert name in DEPENDENT, name


@pytest.mark.parametrize("name", DEPENDENT)
def test_dependent_kernel_waits_and_promises_nothing(name):
    params, body, where = KERNELS[name]
    assert "pdl_wait()" in body, (name, where)
    assert "__restrict__" not in params, (name, where)
    assert not re.search(r"__ldg\s*\(|\bld\.global\.nc\b", body), (name, where)
