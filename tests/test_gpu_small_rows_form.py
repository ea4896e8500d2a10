"""Units of at most 64 query rows can run on more than one tensor-core kernel, and the library picks one by their number
and length (ORTHRUS_TC_SMALL_ROWS, read at every call, overrides it).  The shape, split, edge-case and
in-cache tests run here once with "0", which keeps such units on the kernels for wide ones, and once with "1", which
puts every one of them on the kernel with the keys on the MMA's rows: in a child process, so that
the parity tests themselves need not know of it."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu
HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.mark.parametrize("value", ["0", "1"])
def test_parity_of_the_common_form_on_units_of_at_most_64_rows(value):
    env = dict(os.environ, ORTHRUS_TC_SMALL_ROWS=value)
    r = subprocess.run([sys.executable, "-m", "pytest", os.path.join(HERE, "test_gpu_attend.py"),
                        os.path.join(HERE, "test_gpu_attend_tc_edges.py"),
                        os.path.join(HERE, "test_gpu_truncate_commit.py"), "-x", "-q",
                        "-k", "tcgen05 or edges or cache"],
                       env=env, capture_output=True, text=True, timeout=900)
    assert r.returncode == 0, r.stdout[-3000:] + r.stderr[-2000:]
    assert " passed" in r.stdout
