"""Host plans (mesh, element plan, multigrid hierarchy) where memory or threads
run out: the calls return QPAT_ENOMEM, and no exception of theirs ends the
process.  Each limit runs in a process of its own whose address space is bounded
a little above what it already uses."""
import subprocess
import sys

import pytest

CHILD = r"""
import os, resource, sys
import numpy as np
import qpat_synth as S
import paper_1512_02796_gb300 as Q
xyz, tets = S.kuhn_cube(28, 1.0)
Q.qpat_multigrid_host_info(*S.kuhn_cube(3, 1.0))
used = int(open("/proc/self/statm").read().split()[0]) * os.sysconf("SC_PAGE_SIZE")
resource.setrlimit(resource.RLIMIT_AS, (used + int(sys.argv[1]) * 2**20,) * 2)
for call in (lambda: Q.qpat_multigrid_host_info(xyz, tets), lambda: Q.qpat_mesh_host_info(xyz, tets, 512)):
    try:
        call()
        print("done")
    except Q.QpatError as e:
        assert e.code == -6, e
        print("no memory")
    except MemoryError:
        print("no memory")  # the caller's own arrays
"""


@pytest.mark.parametrize("spare", [2, 8, 16, 24, 32, 48, 64, 96, 128, 192])
def test_plans_without_memory(spare):
    r = subprocess.run([sys.executable, "-c", CHILD, str(spare)], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, (r.returncode, r.stderr[-400:])
    assert r.stdout.split("\n")[0] in ("done", "no memory")
