"""Compiles and loads the tests' own .cu files: launch_rules.cu, the library's host-side
launch rules behind a C interface."""
import ctypes
import functools
import importlib.util
import subprocess
import tempfile
from pathlib import Path

import pytest

ROOT = Path(__file__).resolve().parents[1]
PREC = {"f64": 0, "f32": 1, "f16": 2}


def build_module():
    """the package's build.py, loaded by path"""
    spec = importlib.util.spec_from_file_location("_lbm_build_for_rules", ROOT / "paper_2105_08772_gb300" / "build.py")
    b = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(b)
    return b


@functools.lru_cache(maxsize=None)
def compile_so(source):
    """tests/<source> compiled with the library's flags and loaded"""
    b = build_module()
    try:
        nvcc = b.nvcc()
    except RuntimeError:
        pytest.skip("nvcc not available")
    out = Path(tempfile.mkdtemp(prefix="lbm_tests_")) / (Path(source).stem + ".so")
    cmd = [nvcc, *b.ARCH, *b.NVCC_FLAGS, "-shared", str(ROOT / "tests" / source), "-o", str(out)]
    r = subprocess.run(cmd, capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stderr[-2000:]
    return ctypes.CDLL(str(out))


def batch_mix(prec, stencil, boxes, taus=None, slots=0):
    """(mode, modes that take every box, modes the batch autotuner times) of a set of lattices:
    a group, or a batch of so many slots"""
    n = len(boxes)
    flat = (ctypes.c_int * (3 * n))(*[s for b in boxes for s in b])
    tau = (ctypes.c_double * n)(*(taus or [1.0] * n))
    takes, cand = (ctypes.c_int * 6)(), (ctypes.c_int * 6)()
    mode = compile_so("launch_rules.cu").rule_batch_mix(PREC[prec], stencil, n, flat, tau, slots, takes, cand)
    return mode, {k for k in range(6) if takes[k]}, {k for k in range(6) if cand[k]}


def row_plan(prec, box, sms=152, passes=True):
    """the row kernel's cut of a box as a dict, or None; passes: the lattice has a psi plane"""
    out = (ctypes.c_int * 8)()
    compile_so("launch_rules.cu").rule_row_plan(PREC[prec], *box, sms, int(passes), out)
    keys = ("ok", "aligned", "items", "grid", "by", "zc", "nd", "nc")
    return dict(zip(keys, out)) if out[0] else None


def row_batch_rows(prec, stencil, box):
    return compile_so("launch_rules.cu").rule_row_batch_rows(PREC[prec], stencil, *box)


def row_caps(prec):
    out = (ctypes.c_int * 6)()
    compile_so("launch_rules.cu").rule_row_caps(PREC[prec], out)
    return dict(zip(("slot", "mcap", "kd", "threads", "batch_nd", "batch_nc"), out))


def step_route(prec, box, stencil=4, unit_tau=True, eager=False):
    """what a default step runs: 0 a tile kernel, 1 the row kernel, 2 the two passes"""
    return compile_so("launch_rules.cu").rule_step_route(PREC[prec], stencil, int(unit_tau), *box, int(eager))


def steps_per_graph(route):
    return compile_so("launch_rules.cu").rule_steps_per_graph(route)
