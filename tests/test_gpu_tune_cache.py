"""The autotuner's file (PS_TUNE_CACHE): lines of the present format are applied,
lines written before the schedule's radix chose between tile and Stockham kernels
(one field less) are not, and their geometry is tuned and written again."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CHUNKS = 63  # a choice the tuner never makes
# L1 L2 L3 tile radix ztk ykind xy xfirst chunks tile_x..z radix_x..z + 1
LINE = "20 18 16 {bc} {mode} {sms} 40 36 32 0 1 0 0 0 0 %d 0 0 0 0 0 0" % CHUNKS
CODE = """
from paper_1211_5244_gb300 import psolver
i = psolver.Plan((20, 18, 16), "fff", 0.3, "f32", autotune=True).info()
print("chunks", i.schedule[5])
"""


@pytest.mark.parametrize("suffix,used", [("", False), (" 1", False), (" 2", True)])
def test_old_lines_are_tuned_again(gpu_lib, tmp_path, suffix, used):
    import torch
    from paper_1211_5244_gb300 import psolver
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    mode = psolver.PS_F32 + 4 * (3 * 1 + 2)  # dtype, math 0, order x y z
    free = psolver.PS_BC_FREE
    old = LINE.format(bc="%d %d %d" % (free, free, free), mode=mode, sms=sms)
    line = old + suffix
    path = tmp_path / "tune.txt"
    path.write_text(line + "\n")
    r = subprocess.run([sys.executable, "-c", CODE], cwd=ROOT, capture_output=True, text=True, timeout=300,
                       env=dict(os.environ, PS_TUNE_CACHE=str(path)))
    assert r.returncode == 0, r.stderr
    assert ("chunks %d" % CHUNKS in r.stdout) == used, r.stdout
    lines = path.read_text().splitlines()
    assert lines[0] == line
    if used:
        assert len(lines) == 1
    else:  # the new choice, for the same geometry, in the present format
        assert len(lines) == 2 and lines[1].split()[:8] == line.split()[:8]
        assert len(lines[1].split()) == len(old.split()) + 1 and lines[1].split()[-1] == "2"
