"""The allocation-free step's two ways of reading and writing the caller's order of
the angles (8-byte words and single ones), bitwise against rt_step, and once more
with every index checked (tests/_noalloc_pairs.py)."""
import os
import subprocess
import sys

import pytest

import _noalloc_pairs as np_

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("name,shape,bc,still", np_.CASES, ids=lambda x: "x".join(map(str, x)) if isinstance(x, tuple) else x)
def test_noalloc_pairs_equal_rt_step(name, shape, bc, still):
    np_.rtbuild.build()
    words = np_.words(np_.angle_set(name)[0])
    assert {"all": all(words), "none": not any(words), "some": any(words) and not all(words)}[np_.SETS[name]]
    np_.check(name, shape, bc, still)


def test_no_index_out_of_range_in_the_allocation_free_step():
    r = subprocess.run([sys.executable, os.path.join(np_.HERE, "_noalloc_pairs.py")], capture_output=True, text=True,
                       timeout=1500)
    assert r.returncode == 0 and r.stdout.rstrip().endswith("OK"), (r.stdout[-3000:], r.stderr[-3000:])
