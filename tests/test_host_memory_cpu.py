"""Host memory and threads that run out come back as PHIA_ENOMEM, not as an abort (CPU only: the
address space of a child process is limited after its inputs are made)."""
import os
import subprocess
import sys

from conftest import ROOT

PROGRAM = """
import resource, sys
sys.path.insert(0, %r)
from paper_2407_10205_gb300 import instances as ins
from paper_2407_10205_gb300 import phia
phia.load()
c = ins.erdos_renyi(4000, 0.05, 127, 31, 4, 1)
try:
    phia.create_csr(c.row_ptr[:3], c.col, c.val, c.kh[:2], 4)      # first call's own memory
except phia.PhiaError:
    pass
used = int(open("/proc/self/statm").read().split()[0]) * resource.getpagesize()
codes = set()
for extra in (1, 2, 3, 5, 8, 12, 16, 24, 32):
    resource.setrlimit(resource.RLIMIT_AS, (used + (extra << 20), resource.RLIM_INFINITY))
    try:
        phia.Batch([c, c, c, c])
    except phia.PhiaError as e:
        codes.add(e.code)
    except MemoryError:
        pass
    resource.setrlimit(resource.RLIMIT_AS, (resource.RLIM_INFINITY, resource.RLIM_INFINITY))
print("codes", sorted(codes))
assert phia.ENOMEM in codes
""" % ROOT


def test_no_abort_without_host_memory():
    r = subprocess.run([sys.executable, "-c", PROGRAM], capture_output=True, text=True, env=dict(os.environ, CUDA_VISIBLE_DEVICES=""))
    assert r.returncode == 0, (r.returncode, r.stdout, r.stderr[-800:])
