"""Registers and spills of the row kernels (one CTA of 512 threads per SM: 128 registers
a thread) and of the two-pass kernels (128 threads, as many CTAs as registers allow), from
ptxas's report.  The FP16 row kernels, the FP32 one for aligned rows and all two-pass
kernels spill nothing; the other FP32 row kernels no more than stated beside
kRowThreads."""
import re
import subprocess

import pytest

import launch_rules

KERNEL = re.compile(r"(lattice_row_kernel|lattice_row_batch_kernel)INS_8RowShapeILi(\d)EEELb([01])E"
                    r"|(split_moments_kernel|split_collide_kernel)I([df])(?:Li(\d)ELb([01]))?")
F32, F16 = "1", "2"
SPILL = {("lattice_row_kernel", F32, "0"): 12, ("lattice_row_batch_kernel", F32, "1"): 24,
         ("lattice_row_batch_kernel", F32, "0"): 52}


@pytest.fixture(scope="module")
def report(tmp_path_factory):
    b = launch_rules.build_module()
    try:
        nvcc = b.nvcc()
    except RuntimeError:
        pytest.skip("nvcc not available")
    tmp = tmp_path_factory.mktemp("ptxas")
    jobs = [subprocess.Popen([nvcc, *b.ARCH, *b.NVCC_FLAGS, "-Xptxas", "-v", "-c", str(src), "-o", str(tmp / (src.stem + ".o"))],
                             stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True)
            for src in (b.CSRC / "lbm_row.cu", launch_rules.ROOT / "tests" / "split_kernels.cu")]
    out, key, spill = {}, None, 0
    for job in jobs:
        text = job.communicate(timeout=900)[0]
        assert job.returncode == 0, text[-2000:]
        for line in text.splitlines():
            if "Compiling entry function" in line:
                m = KERNEL.search(line)
                key = tuple(g for g in m.groups() if g is not None) if m else None
            elif key and "bytes spill stores" in line:
                spill = int(re.search(r"(\d+) bytes spill stores", line).group(1))
            elif key and "Used" in line:
                out[key] = (int(re.search(r"Used (\d+) registers", line).group(1)), spill)
                key = None
    return out


def test_row_kernels(report):
    rows = {k: v for k, v in report.items() if k[0].startswith("lattice_row")}
    assert len(rows) == 6, sorted(report)
    for key, (regs, spill) in rows.items():
        assert regs <= 128 and spill <= SPILL.get(key, 0), (key, regs, spill)


def test_two_pass_kernels(report):
    split = {k: v for k, v in report.items() if k[0].startswith("split")}
    assert len(split) == 14, sorted(report)
    for key, (regs, spill) in split.items():
        assert regs <= 128 and spill == 0, (key, regs, spill)
