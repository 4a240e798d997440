"""Memory safety of the kernels' larger and rarer forms, as the small-lattice
battery has it for the others: every form of the on-chip warp, the band kernel,
one and several clusters, both layouts' half-sweeps, the planned random words and
the packing, against the build that checks indices instead of using bad ones."""
import json
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_forms_under_the_checked_build():
    from paper_1811_04384_gb300 import build
    env = dict(os.environ, ISING_LIBRARY=build.build(checked=True))
    r = subprocess.run([sys.executable, os.path.join(ROOT, "tests", "helpers", "checked_forms.py")],
                       capture_output=True, text=True, env=env, timeout=900)
    assert r.returncode == 0, r.stdout[-2000:] + r.stderr[-2000:]
    out = json.loads(r.stdout.strip().splitlines()[-1])
    assert out["ok"] and out["checked"] and out["violation"] == 0
    assert out["cases"] >= 40
