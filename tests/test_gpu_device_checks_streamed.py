"""Device index checks of the streamed kernels, of resident launches of large and wide runs and of MRCA
samples of several blocks: the device-check build tests every global index and records GA_EBOUNDS
instead of making an out-of-range access.  Every status must stay clean and every result equal the
oracle's."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))


def test_no_index_check_fails_streamed():
    from paper_2405_03605_gb300 import build
    lib = build.build(debug=True)
    env = dict(os.environ, PAPER_2405_03605_GB300_LIB=lib)
    res = subprocess.run([sys.executable, os.path.join(HERE, "device_checks_streamed_worker.py")],
                         env=env, capture_output=True, text=True, timeout=900)
    assert res.returncode == 0, res.stdout[-2000:] + res.stderr[-4000:]
    assert "device checks clean" in res.stdout
