"""The bounds-checking debug library over the kernels of N' = 4096 and 8192 in
FP32 and over dense tiles of bright and faint samples."""
import json
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_no_access_of_the_largest_passes_leaves_its_buffer():
    from paper_1308_6644_gb300 import _build
    lib = _build.build_debug()
    env = dict(os.environ, NUASM_LIBRARY=lib)
    r = subprocess.run([sys.executable, os.path.join(ROOT, "tests", "debug_bounds_large_run.py")], env=env,
                       capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stderr[-3000:]
    records = json.loads(r.stdout.strip().splitlines()[-1])
    assert len(records) == 10
    bad = [rec for rec in records if rec["hits"] != 0]
    assert not bad, bad
