"""The batched engine (queue entries, late decisions, sigma fields) under the debug
build's index checks and guard bands."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_batched_queue_suite_passes_the_debug_checks():
    sys.path.insert(0, ROOT)
    from paper_2006_16465_gb300 import _build
    _build.build(debug=True)
    r = subprocess.run([sys.executable, "-m", "pytest", "tests/test_gpu_batched_queue.py", "tests/test_gpu_batched_sizes.py",
                        "-m", "gpu", "-q", "-p", "no:cacheprovider", "-x"],
                       cwd=ROOT, env=dict(os.environ, HJ_LIBRARY="debug"), capture_output=True, text=True, timeout=1800)
    tail = "\n".join(r.stdout.splitlines()[-15:])
    assert r.returncode == 0, tail + r.stderr[-2000:]
    assert " passed" in tail
