"""How the kernels that may be resident before their operand is complete read
it (CPU only, from the sources).  A kernel launched by srt_launch starts with
srt_in_order(), which waits for the kernel before; until then that kernel may
still write the operand, so it must be read by plain loads that the compiler
cannot move above the wait (the volatile srt_ld_* helpers of common.cuh), and
never as read-only data."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2402_15641_gb300", "csrc")


def _source(path):
    s = open(path).read()
    s = re.sub(r"/\*.*?\*/", "", s, flags=re.S)
    return re.sub(r"//[^\n]*", "", s)


def _body(s, start):
    """Text of the braces that open at or after start."""
    i = s.index("{", start)
    depth = 0
    for k in range(i, len(s)):
        depth += {"{": 1, "}": -1}.get(s[k], 0)
        if depth == 0:
            return s[i + 1:k]
    raise AssertionError("unbalanced braces")


def _kernels(early):
    """(file, kernel, operand parameter, body) of every kernel that waits for
    the one before (early) or of every other."""
    out = []
    for f in sorted(glob.glob(os.path.join(CSRC, "*.cu"))):
        s = _source(f)
        for m in re.finditer(r"__global__[^;{]*?\b(k_\w+)\(([^{;]*?)\)\s*\{", s):
            body = _body(s, m.end() - 1)
            if ("srt_in_order" in body) == early:
                operand = re.findall(r"const float\*\s*(?:__restrict__)?\s*(\w+)", m.group(2))
                out.append((os.path.basename(f), m.group(1), operand, body))
    return out


def test_every_early_kernel_is_found():
    early = {k for _, k, _, _ in _kernels(True)}
    assert early == {"k_rows", "k_tile22", "k_a1t_tile", "k_a1t_split", "k_transpose", "k_transpose_v4"}
    # the others are launched in order, by <<< >>>, and these never are
    for f in glob.glob(os.path.join(CSRC, "*.cu")):
        s = _source(f)
        plain = set(re.findall(r"\b(k_\w+)(?:<[^;<>]*>)?\s*<<<", s))
        assert not plain & early, f
        for name in set(re.findall(r"__global__[^;{]*?\b(k_\w+)\(", s)) - early:
            assert name in plain, name


@pytest.mark.parametrize("file,kernel,operand,body", _kernels(True), ids=lambda v: v if isinstance(v, str) and
                         len(v) < 20 else "")
def test_waits_first_and_reads_its_operand_behind_the_wait(file, kernel, operand, body):
    assert body.lstrip().startswith("srt_in_order();")
    assert len(operand) == 1
    # names that hold addresses of the operand: x, then x0 = x + .., xr = x0 + ..
    names = set(operand)
    for _ in range(3):
        for name, value in re.findall(r"const float\*\s*(\w+)\s*=\s*([^;]*);", body):
            if any(re.search(rf"\b{n}\b", value) for n in names):
                names.add(name)
    for n in names:
        assert not re.search(rf"__ldg\([^;]*\b{n}\b", body), n
        assert not re.search(rf"\b{n}\s*\[", body), n
        assert not re.search(rf"(^|[=(,{{;?:])\s*\*\s*{n}\b", body), n


def test_no_read_only_load_in_the_operand_helpers():
    for f in glob.glob(os.path.join(CSRC, "*.cu*")):
        assert "ld.global.nc" not in _source(f), f
    s = _source(os.path.join(CSRC, "common.cuh"))
    for name in ("srt_ld_keep", "srt_ld4", "srt_ld2", "srt_ld1"):
        b = _body(s, s.index(name))
        assert "asm volatile(" in b and "ld.global" in b and ".nc" not in b
    rows = _source(os.path.join(CSRC, "spmm.cu"))
    assert "__ldg" not in _body(rows, rows.index("ld_cols("))
