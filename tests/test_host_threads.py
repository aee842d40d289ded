"""Host work on several threads: every item once, an item's exception thrown to
the caller after the others have run, and the same where the system starts no
further thread (address space too small for a thread's stack), which must not
end the process."""
import os
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = """
import resource, sys
import numpy as np
from paper_2009_01287_gb300 import binding
L = binding.inspect_lib()
done = np.zeros(500, dtype=np.int32)
if sys.argv[1] == "few":
    used = int(open("/proc/self/statm").read().split()[0]) * resource.getpagesize()
    resource.setrlimit(resource.RLIMIT_AS, (used + (4 << 20), resource.RLIM_INFINITY))
    import threading
    try:
        threading.Thread(target=lambda: None).start()
        sys.exit(7)   # threads still start: nothing shown
    except RuntimeError:
        pass
for fails in (-1, 0, 499):
    done[:] = 0
    assert L.dginspect_on_threads(500, fails, done.ctypes.data) == (fails >= 0)
    assert (done == 1).all()
"""


@pytest.mark.parametrize("threads", ["many", "few"])
def test_every_item_once(built_lib, threads):
    r = subprocess.run([sys.executable, "-c", PROGRAM, threads], cwd=ROOT, capture_output=True, text=True)
    if r.returncode == 7:
        pytest.skip("this system starts threads in any address space")
    assert r.returncode == 0, r.stderr
