"""A SLICE4 context that the device has no room for (J^(q), K^(q) of 8192 functions and orbitals would
take 9 TB): E_OOM, without host memory spent on the unit lists of a problem that cannot be."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
import resource
import numpy as np
from types import SimpleNamespace
from paper_2012_15662_gb300 import binding as bd
from synthetic import make_system, pairing_columns

bd.Engine(make_system("square"), bd.DONOF_RI_SLICE4).close()  # the library and the device's context
n = 8192
sub, rank = pairing_columns(n // 2, 1)
s = SimpleNamespace(atom_xyz=np.zeros((1, 3)), atom_charge=np.ones(1), bf_atom=np.zeros(n, np.int32),
                    bf_alpha=np.linspace(0.1, 10.0, n), aux_atom=np.zeros(1, np.int32), aux_alpha=np.ones(1),
                    n_strong=n // 2, n_weak_per=1)
before = resource.getrusage(resource.RUSAGE_SELF).ru_maxrss
try:
    bd.donof_ri_init(s, sub, rank, bd.DONOF_RI_SLICE4)
    status = 0
except bd.DonofError as e:
    status = e.status
print(status, resource.getrusage(resource.RUSAGE_SELF).ru_maxrss - before)
"""


def test_host_memory_of_a_context_that_does_not_fit():
    out = subprocess.run([sys.executable, "-c", PROGRAM], cwd=ROOT, capture_output=True, text=True, check=True, timeout=600)
    status, grown_kb = map(int, out.stdout.split())
    assert status == -2
    assert grown_kb < 200 * 1024
