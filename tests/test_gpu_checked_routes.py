"""The bounds-checked build over split, ring, prefetching and column-merge launches
(needs a GPU): checked_routes.py in a process of its own, no failed check."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_checked_routes_have_no_failed_checks():
    from paper_2501_10653_gb300 import build
    lib = build.build(checked=True)
    env = dict(os.environ, IQA_LIBRARY=lib,
               PYTHONPATH=os.pathsep.join([os.path.join(ROOT, "tests"), ROOT,
                                           os.environ.get("PYTHONPATH", "")]))
    r = subprocess.run([sys.executable, "-c", "import checked_routes; checked_routes.main()"],
                       cwd=ROOT, env=env, capture_output=True, text=True, timeout=900)
    assert r.returncode == 0, r.stdout[-3000:] + r.stderr[-3000:]
    assert "checked routes: no failed checks" in r.stdout
