"""Threads that share a stream share the scratch memory of the binding: their calls are enqueued one after the other, while
calls on different streams may be enqueued side by side."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_calls_of_several_threads_on_one_stream_do_not_mix():
    env = dict(os.environ, PYTHONPATH=ROOT + os.pathsep + os.environ.get("PYTHONPATH", ""))
    res = subprocess.run([sys.executable, "-m", "tests._binding_threads_worker"], cwd=ROOT, env=env, capture_output=True,
                         text=True, timeout=300)
    assert res.returncode == 0, res.stdout[-2000:] + res.stderr[-2000:]
    assert "at once: 1 on a stream, 2 in all" in res.stdout, res.stdout
