"""The checked build over both forms of the bank render (checked_render.py): no failed index check, and
bitwise the normal build's outputs."""
import json
import os
import subprocess
import sys

import pytest

import checked_render

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_checked_renders(sdlib):
    subprocess.run([sys.executable, "-c",
                    "from paper_2503_11213_gb300 import build as b; b.build(checked=True)"],
                   cwd=ROOT, check=True)
    r = subprocess.run([sys.executable, os.path.join(ROOT, "tests", "checked_render.py")], cwd=ROOT,
                       env=dict(os.environ, SDIRT_CHECKED="1"), capture_output=True, text=True,
                       timeout=900)
    assert r.returncode == 0, r.stderr[-3000:]
    res = json.loads(r.stdout.strip().splitlines()[-1])
    assert res["count"] == 0 and res["site"] == 0, res
    assert res["hashes"] == checked_render.run(sdlib)
