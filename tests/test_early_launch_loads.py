"""Kernels that may be put in place early (pdl_enter) overlap the kernel before, whose output they read: no
load of that may take the read-only path, which is for memory that nobody writes while the kernel lives.  The
read-only load (ld_old) is kept for what is written two or more kernels before any reader."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1912_00323_gb300", "csrc")


def _code(name):
    with open(os.path.join(CSRC, name)) as f:
        return re.sub(r"//[^\n]*|/\*.*?\*/", "", f.read(), flags=re.S)


EARLY = sorted(f for f in os.listdir(CSRC) if f.endswith((".cu", ".cuh")) and "pdl_enter();" in _code(f))


def test_files_found():
    assert {"cells.cuh", "hd_kernels.cuh", "lowd_kernels.cuh", "sort.cu", "tc_kernels.cuh"} <= set(EARLY)


@pytest.mark.parametrize("name", EARLY)
def test_no_read_only_loads(name):
    src = _code(name)
    assert "__ldg(" not in src and "ld.global.nc" not in src
    assert set(re.findall(r"const\s+[\w:<>, ]+\*\s*__restrict__\s*(\w+)", src)) <= {"in"}
    # the input and its gathered rows (or a pointer into them), the sets' tables, the lists of points
    read = set(re.findall(r"ld_old\((?:reinterpret_cast<[^>]*>\()?\(?([\w.]+)", src))
    assert read <= {"in", "src", "p", "a", "b", "pts", "mm", "set_off", "tt.row_list", "tt.core_list", "tt.nc_list"}


@pytest.mark.parametrize("name", EARLY)
def test_early_kernels_wait_first(name):
    """Every kernel given to launch() in these files starts with pdl_enter()."""
    src = _code(name)
    for m in re.finditer(r"__global__[^;{]*?\b(k_\w+)\s*\(", src):
        depth, j = 1, m.end()
        while depth:
            depth += {"(": 1, ")": -1}.get(src[j], 0)
            j += 1
        assert src[src.index("{", j) + 1:].lstrip().startswith("pdl_enter();"), m.group(1)


def test_mail_number_is_released():
    """The host takes the mailbox's words when it sees the number: the thread that stores the number fences at
    system scope after the block's barrier."""
    src = _code("lowd_kernels.cuh")
    body = src[src.index("k_mail("):src.index("*number = value")]
    after = body[body.rindex("__syncthreads();"):]
    assert "if (threadIdx.x == 0)" in after and "__threadfence_system();" in after
