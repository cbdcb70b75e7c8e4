"""Source checks of the kernels that start before the kernel ahead of them in
the stream has finished (launch_pdl; CPU only: a stale read would be a race).
Such a kernel is resident while its inputs are still being written, so it must
not read them through the read-only path (__ldg, or a plain read of a const
__restrict__ pointer, which the compiler may turn into one), and it must wait
before it reads them."""
import os
import re
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2605_31481_gb300", "csrc")


def _read(name):
    with open(os.path.join(CSRC, name)) as fh:
        return re.sub(r"//[^\n]*", "", fh.read())


def _units():
    return [f for f in sorted(os.listdir(CSRC)) if f.endswith(".cu") and "launch_pdl(" in _read(f)]


def _braced(src, at):
    """The text from the brace at or after `at` to its match."""
    start = at = src.index("{", at)
    depth = 0
    while True:
        depth += {"{": 1, "}": -1}.get(src[at], 0)
        at += 1
        if depth == 0:
            return src[start:at]


def _waits(src):
    """The macros of a unit that hold the wait."""
    text = src.replace("\\\n", " ")
    macros = dict(re.findall(r"#define (\w+)(?:\([^)]*\))?([^\n]*)", text))
    names, grown = {"pdl_wait()"}, True
    while grown:
        more = {n for n, body in macros.items() if any(w in body for w in names)} - names
        names |= more
        grown = bool(more)
    return names


def _kernels():
    """(unit, name, parameters, body) of every kernel of these units that waits for the one ahead."""
    out = []
    for unit in _units():
        src = _read(unit)
        waits = _waits(src)
        for m in re.finditer(r"__global__ void (?:__launch_bounds__\([^)]*\)\s*)?(\w+)\(", src):
            body = _braced(src, m.end())
            if any(w in body for w in waits):
                out.append((unit, m.group(1), src[m.end():src.index("{", m.end())], body))
    return out


def test_the_kernels_are_found():
    names = {k[1] for k in _kernels()}
    assert {"partial_reduce_kernel", "wb_vjp_kernel", "wb_aba_vjp_kernel", "rnea_vjp_lean_kernel", "fk_vjp_tile_kernel",
            "aba_lean_kernel", "crba_lean_kernel", "eval_tile_kernel", "multi_tile_kernel"} <= names


def test_no_read_only_loads_behind_the_wait():
    kernels = _kernels()
    for unit, name, params, body in kernels:
        assert "__ldg(" not in body, (unit, name)
        for p in re.findall(r"const float\*\s*__restrict__ (\w+)", params):
            assert not re.search(rf"(?<![\w.]){p}\s*\[|\*\s*{p}\b(?!\s*\+)", body), (unit, name, p)
    # the device code of units in which every kernel is launched that way
    for unit in {k[0] for k in kernels}:
        header = unit.replace(".cu", ".cuh")
        n_kernels = len(re.findall(r"__global__ void", _read(unit)))
        if os.path.exists(os.path.join(CSRC, header)) and n_kernels == sum(k[0] == unit for k in kernels):
            assert "__ldg(" not in _read(header), header
    assert "__ldg(" not in _read("level.cuh")


def test_every_kernel_waits_before_it_stages_inputs():
    for unit, name, _, body in _kernels():
        first = re.search(r"stage_block_rows|ld_input|vjp_warp|minv_warp|rnea_vjp_lean\(", body)
        wait = min((body.index(w) for w in _waits(_read(unit)) if w in body))
        assert first is None or wait < first.start(), (unit, name)


def test_a_refused_launch_leaves_no_error_behind(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("needs nvcc")
    root = os.path.dirname(os.path.dirname(CSRC))
    exe = tmp_path / "launch_errors"
    host = os.path.join(root, "tests", "host", "launch_errors")
    cmd = [nvcc, "-std=c++17", "-cudart", "none", "-I", CSRC, "-I", os.path.join(root, "include"), host + ".cu",
           host + ".cpp", "-o", str(exe)]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-3000:]
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0 and r.stdout.strip() == "ok", r.stdout + r.stderr
