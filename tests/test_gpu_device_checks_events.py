"""The event-driven sweep under the checked build (tests/checked_events.py):
results equal the oracle's, no index leaves its array and no distance comes
from shared memory that nothing wrote (the checked build fills it with negative
numbers first; distances are not negative)."""
import json
import os
import subprocess
import sys

import pytest

from conftest import has_gpu
from paper_2608_25376_gb300 import build as qbuild

pytestmark = pytest.mark.gpu
HERE = os.path.dirname(os.path.abspath(__file__))


def test_checked_event_sweep():
    if not has_gpu():
        pytest.skip("no CUDA device")
    env = dict(os.environ, QPATH_LIBRARY=qbuild.build(checked=True))
    r = subprocess.run([sys.executable, os.path.join(HERE, "checked_events.py")], env=env, capture_output=True,
                       text=True, timeout=1200)
    assert r.returncode == 0, r.stdout[-3000:] + r.stderr[-4000:]
    line = json.loads(r.stdout.strip().splitlines()[-1])
    assert line["enabled"] and line["first_failure"] == 0 and all(v is True for v in line["results"].values())
