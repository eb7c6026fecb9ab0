"""Rules of the inline PTX that no run on a device shows: checked on the
sources, and on the host path of the helpers (no GPU needed)."""
import glob
import os
import re
import subprocess

import pytest

from test_native_helpers import HERE, nvcc

CSRC = os.path.join(HERE, os.pardir, "paper_2208_11447_gb300", "csrc")


def sources():
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        with open(path) as f:
            yield os.path.basename(path), f.read()


def test_policy_fractions_lie_in_range(tmp_path):
    """createpolicy.fractional is defined for fractions in (0, 1] only."""
    assigned = [m.strip() for _, text in sources() for m in re.findall(r"\bl2_frac\s*=\s*([^;]*);", text)]
    assert assigned and all(re.fullmatch(r"l2_keep_fraction\([^?]*\)", a) for a in assigned), assigned
    exe = nvcc()
    if exe is None:
        pytest.skip("nvcc not found")
    out = str(tmp_path / "l2_fraction")
    res = subprocess.run([exe, "-std=c++17", "-O2", "-o", out, os.path.join(HERE, "native", "l2_fraction.cu")],
                         capture_output=True, text=True)
    assert res.returncode == 0, res.stderr
    run = subprocess.run([out], capture_output=True, text=True, timeout=120)
    assert run.returncode == 0, run.stdout + run.stderr



def test_statements_that_access_memory_say_so():
    """A statement that stores, or adds to memory, through an address the
    compiler does not see carries the "memory" clobber: the sketch bins are
    cleared and read by ordinary accesses on both sides."""
    found, bare = 0, []
    for name, text in sources():
        for m in re.finditer(r"asm\s+volatile\s*\(((?:[^;\"]|\"[^\"]*\")*)\)\s*;", text):
            if re.search(r"\"\s*(red|st|atom)\.", m.group(1)):
                found += 1
                if '"memory"' not in m.group(1):
                    bare.append((name, m.group(1)))
    assert found > 0 and not bare, bare
