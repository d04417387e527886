"""Registers and spills of the score and team kernels, as the compiler reports them
(CPU only: nvcc cross-compiles two map formats' translation units)."""
import os
import re
import subprocess

import pytest

from test_kernel_registers_cpu import CSRC, ROOT, _nvcc


@pytest.mark.slow
def test_score_and_team_kernels_keep_their_budgets(tmp_path):
    """Score kernels (atoms per lane, many conformations or one per scheduler): no spills
    within the registers that their warps per SM leave.  Team kernels (CTAs of eight
    warps per SM, tiles): one atom per lane without spills."""
    nvcc = _nvcc()
    if nvcc is None:
        pytest.skip("nvcc not found")
    procs = {}
    for fmt in (0, 3, 4):
        cmd = [nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-O3", "-std=c++17", "-Xptxas", "-v",
               "-I", os.path.join(ROOT, "include"), "-I", CSRC, "-c", os.path.join(CSRC, f"dock_fmt{fmt}.cu"),
               "-o", str(tmp_path / f"dock_fmt{fmt}.o")]
        procs[fmt] = subprocess.Popen(cmd, stdout=subprocess.PIPE, stderr=subprocess.PIPE, text=True)
    score_limit = {(1, 0): 96, (2, 0): 80, (1, 1): 128, (2, 1): 128}
    for fmt, proc in procs.items():
        _, err = proc.communicate(timeout=900)
        assert proc.returncode == 0, err[-2000:]
        found = {}
        for name, spill, regs in re.findall(
                r"Compiling entry function '(\S+)'.*?(\d+) bytes spill stores.*?Used (\d+) registers", err, re.S):
            found[name] = (int(spill), int(regs))
        score = {tuple(map(int, m.groups())): v for n, v in found.items()
                 if (m := re.search(r"score_eval_kernelILi(\d)ELi%dELb(\d)E" % fmt, n))}
        team = {tuple(map(int, m.groups())): v for n, v in found.items()
                if (m := re.search(r"dock_team_kernelILi%dELi(\d)ELi(\d)E" % fmt, n))}
        assert set(score) == set(score_limit) and set(team) == {(1, 1), (1, 3), (2, 1), (2, 3)}
        for key, (spill, regs) in score.items():
            assert spill == 0 and regs <= score_limit[key], (fmt, key, spill, regs)
        for key, (spill, regs) in team.items():
            assert regs <= (128 if key[0] == 2 else 255), (fmt, key, regs)
            assert spill == 0 or key == (2, 3), (fmt, key, spill)
