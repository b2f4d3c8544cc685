"""The kernels' shared-memory limits are attributes of a device: a process that
makes handles on several GPUs raises them on each.  Checked on the CPU against a
stand-in for the CUDA runtime's calls, whose allocations fail, so that kmc_create
ends with KMC_E_NOMEM after it has set the limits and before it would launch."""
import os
import shutil
import subprocess
import sys

import pytest

from paper_2511_09413_gb300 import build

FAKE = r"""
#include <stddef.h>
static int dev, count[4], fail;
void fake_device(int d) { dev = d; }
void fake_fail(int f) { fail = f; }
int fake_count(int d) { return count[d]; }
int cudaGetDevice(int *d) { *d = dev; return 0; }
int cudaFuncSetAttribute(const void *f, int a, int v) { count[dev] += 1; return fail; }
int cudaMallocAsync(void **p, size_t n, void *s) { return 2; }
int cudaFreeAsync(void *p, void *s) { return 0; }
int cudaStreamSynchronize(void *s) { return 0; }
int cudaGetLastError(void) { return 0; }
"""

USE = r"""
import ctypes, sys
import numpy as np
from paper_2511_09413_gb300 import kmc as K
fake = ctypes.CDLL(sys.argv[1])
p = K.kmc_params(n_rails=4, n_sites=100, n_zones=10, site_spacing_nm=1.0, dt_s=1e-9, T_K=300.0, Ea_eV=0.4,
                 nu_Hz=1e12, alpha_V=0.2, kappa=1.0, init_mode=1, fill=0.2)
def create(code):
    try:
        K.kmc_create(p, np.zeros(3))
    except K.KmcError as e:
        assert e.code == code, str(e)
    else:
        raise AssertionError("created")
create(K.KMC_E_NOMEM)
once = fake.fake_count(0)
assert once > 0
create(K.KMC_E_NOMEM)
assert fake.fake_count(0) == once               # once a device
fake.fake_device(2)
create(K.KMC_E_NOMEM)
assert fake.fake_count(2) == once, fake.fake_count(2)
fake.fake_device(1)
fake.fake_fail(1)                               # a limit that cannot be raised is tried again
create(K.KMC_E_CUDA)
fake.fake_fail(0)
create(K.KMC_E_NOMEM)
assert fake.fake_count(1) > once
"""


@pytest.mark.skipif(not shutil.which("gcc"), reason="gcc not available")
def test_limits_are_raised_on_every_device(tmp_path):
    build.build()
    src, so = tmp_path / "fake.c", tmp_path / "libfake.so"
    src.write_text(FAKE)
    subprocess.run(["gcc", "-shared", "-fPIC", "-o", str(so), str(src)], check=True)
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", USE, str(so)], cwd=root, capture_output=True, text=True,
                       env=dict(os.environ, LD_PRELOAD=str(so)), timeout=300)
    assert r.returncode == 0, r.stderr
