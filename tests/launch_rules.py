"""Loads the library's host-side launch rules (launch_rules.cu) for the CPU tests."""
import ctypes
import functools
import importlib.util
import subprocess
import tempfile
from pathlib import Path

import pytest

ROOT = Path(__file__).resolve().parents[1]
PREC = {"f64": 0, "f32": 1, "f16": 2}


@functools.lru_cache(maxsize=None)
def load():
    spec = importlib.util.spec_from_file_location("_lbm_build_for_rules", ROOT / "paper_2105_08772_gb300" / "build.py")
    b = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(b)
    try:
        nvcc = b.nvcc()
    except RuntimeError:
        pytest.skip("nvcc not available")
    out = Path(tempfile.mkdtemp(prefix="launch_rules_")) / "rules.so"
    cmd = [nvcc, *b.ARCH, *b.NVCC_FLAGS, "-shared", str(ROOT / "tests" / "launch_rules.cu"), "-o", str(out)]
    r = subprocess.run(cmd, capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stderr[-2000:]
    return ctypes.CDLL(str(out))


def batch_mix(prec, stencil, boxes, taus=None):
    """(mode, modes that take every box, modes the batch autotuner times) of a set of lattices"""
    n = len(boxes)
    flat = (ctypes.c_int * (3 * n))(*[s for b in boxes for s in b])
    tau = (ctypes.c_double * n)(*(taus or [1.0] * n))
    takes, cand = (ctypes.c_int * 6)(), (ctypes.c_int * 6)()
    mode = load().rule_batch_mix(PREC[prec], stencil, n, flat, tau, takes, cand)
    return mode, {k for k in range(6) if takes[k]}, {k for k in range(6) if cand[k]}
