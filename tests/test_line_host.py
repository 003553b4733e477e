"""The arithmetic that the double-float FFT lines run (csrc/adp.cuh), compiled for the CPU
and run in the lines' own stage schedules against a direct 80-bit DFT (no GPU).

What it pins, for uniform, constant, spiky, eight-decade, alternating, single-tone, low-part
and largest-sum inputs:
  - the grid invariants: at an aligned stage's input every high part is at most 2^HEAD
    quanta (19; 18 with 16 points per thread and in mixed lines), at its output below 2^23
    quanta and on the grid, so that every sum was exact;
  - the error: below 2^-37 of L times the input bound, and in mixed lines no more than the
    same schedule leaves after an exact first stage. The first stage's own rounding adds at
    most 12 roundings of 2^-47 on sums of R sqrt(2) times the bound (in chains no longer than
    a radix-9 butterfly's), over L: 12 sqrt(2) 2^-47 = 1.2e-13. The later stages round
    other values after it, so their error is drawn anew: 1.5 covers the spread of a
    line's largest error over the mean of 8 inputs.
"""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_1308_0730_gb300", "csrc")
INCLUDE = os.path.join(os.path.dirname(HERE), "include")


@pytest.fixture(scope="module")
def exe(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not found")
    out = str(tmp_path_factory.mktemp("line") / "line_host_check")
    cmd = [nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-O2", "-std=c++17", "--expt-relaxed-constexpr",
           "-Xcompiler", "-ffp-contract=off", "-I", CSRC, "-I", INCLUDE,
           os.path.join(HERE, "native", "line_host_check.cu"), "-o", out]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    return out


@pytest.mark.parametrize("mode", ["regs", "mixed"])
def test_line_schedules_against_80_bit_dft(exe, mode):
    r = subprocess.run([exe, mode], capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stderr
    rows = [line.split() for line in r.stdout.strip().splitlines()]
    assert len(rows) == 8 * (9 if mode == "regs" else 14)
    for plan, pat, err, ref, head, out, on_grid in rows:
        what = f"length:radix {plan}, pattern {pat}"
        most = 19 if mode == "regs" and plan.endswith(":8") else 18
        assert float(head) <= most, f"{what}: a stage input reached 2^{head} q"
        assert float(out) < 23 and on_grid == "1", f"{what}: a sum left the grid (outputs up to 2^{out} q)"
        assert float(err) < 2.0 ** -37, f"{what}: error {float(err):.3e} of L x bound"
        if mode == "mixed":
            assert float(err) <= 1.5 * float(ref) + 12 * 2 ** 0.5 * 2.0 ** -47, f"{what}: {err} against {ref}"
