"""Registers of the kernels whose speed rests on the CTAs that share an SM: as
the compiler reports them for the build's own command line, without spills
(65,536 registers per SM, given out in eights per thread)."""
import re
import subprocess

import pytest

from paper_2407_07253_gb300 import build as B

# object file, kernel: threads per CTA, CTAs per SM
WANT = {
    ("kernels.o", "gj_inverse_globalE"): (512, 4),      # all of an SM's threads
    ("kernels.o", "saddle_inverse_smemE"): (256, 5),    # the 41 KB of a P4 star leave room for five
    ("stokes_mg.o", "pull_scatterIdLb0ELi4"): (256, 8),  # large levels in FP64: gathers in flight
    ("stokes_mg.o", "pull_scatterIdLb0ELi8"): (256, 5),
    ("stokes_mg.o", "pull_scatterIfLb.ELi8"): (256, 8),
}


@pytest.fixture(scope="module")
def reports(tmp_path_factory):
    out = tmp_path_factory.mktemp("ptxas")
    jobs = {o: subprocess.Popen(B._sources()[o] + ["-Xptxas", "-v", "-o", str(out / o)], stderr=subprocess.PIPE, text=True)
            for o in sorted({o for o, _ in WANT})}
    text = {o: j.communicate()[1] for o, j in jobs.items()}
    assert not any(j.returncode for j in jobs.values())
    return text


@pytest.mark.parametrize("obj,name", sorted(WANT))
def test_ctas_per_sm(reports, obj, name):
    threads, ctas = WANT[obj, name]
    found = re.findall(r"entry function '_ZN5skern\d+%s\S*' for .*\n.*\n.*, (\d+) bytes spill stores.*\n.*Used (\d+) registers"
                       % name, reports[obj])
    assert found
    for spilled, regs in found:
        assert int(spilled) == 0
        assert 65536 // ((int(regs) + 7) // 8 * 8 * threads) >= ctas, regs
