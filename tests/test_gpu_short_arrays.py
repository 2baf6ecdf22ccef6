"""Device arrays shorter than a call needs are refused on the host, not read or
written out of range by a kernel (tests/_short_array_child.py)."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.mark.parametrize("length", ["exact", "short"])
@pytest.mark.parametrize("call", ["material", "intensity", "moments", "sources"])
def test_array_shorter_than_the_call_needs(call, length):
    r = subprocess.run([sys.executable, os.path.join(HERE, "_short_array_child.py"), call, length], capture_output=True,
                       text=True, timeout=300)
    assert r.returncode == 0 and r.stdout.rstrip().endswith("OK"), (r.stdout[-2000:], r.stderr[-2000:])
