"""Registers of the kernels whose speed rests on the CTAs that share an SM: as
the compiler reports them for the build's own command line, without spills
(65,536 registers per SM, given out in eights per thread)."""
import re
import subprocess

import pytest

from paper_2407_07253_gb300 import build as B

# kernel: threads per CTA, CTAs per SM
WANT = {
    "gj_inverse_global": (512, 4),      # all of an SM's threads
    "saddle_inverse_smem": (256, 5),    # the 41 KB of a P4 star leave room for five
}


@pytest.fixture(scope="module")
def report(tmp_path_factory):
    cmd = B._sources()["kernels.o"] + ["-Xptxas", "-v", "-o", str(tmp_path_factory.mktemp("ptxas") / "kernels.o")]
    return subprocess.run(cmd, capture_output=True, text=True, check=True).stderr


@pytest.mark.parametrize("name", sorted(WANT))
def test_ctas_per_sm(report, name):
    threads, ctas = WANT[name]
    m = re.search(r"entry function '_ZN5skern\d+%sE\S*' for .*\n.*\n.*, (\d+) bytes spill stores.*\n.*Used (\d+) registers"
                  % name, report)
    assert int(m[1]) == 0
    assert 65536 // ((int(m[2]) + 7) // 8 * 8 * threads) >= ctas, m[0]
