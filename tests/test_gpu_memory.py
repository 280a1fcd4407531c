"""Requests in little device memory: what fitted with the fewest state blocks still fits, and a call made twice takes
the same route both times.  Each case runs in a process of its own, which first fills the device but for the stated
number of megabytes (the library's pool then has exactly that to grow into)."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PRELUDE = """
import sys
sys.path.insert(0, {root!r})
import numpy as np, torch
import __graft_entry__
__graft_entry__.build()
from paper_2510_17432_gb300 import capi
S = capi.request
ctx = capi.tbpm_create(0)
small = capi.tbpm_lattice_create(ctx, capi.lattice_desc(1, (64, 40), t=-2.7, W=1.0, seed=3, vacancy_frac=0.1))
E = np.array([-1.0, 0.3])
def warm():  # kernels loaded before the memory is counted
    capi.tbpm_moments(ctx, small, S(n_states=4, n_moments=64), np.zeros((4, 64, 2)))
    capi.tbpm_conductivity(ctx, small, S(n_states=1, form=2, n_steps=4, time_block=2), 0, E,
                           np.zeros((1, 2, 5), np.complex128), np.zeros((1, 2)))
warm()
def fill(mb):
    free = torch.cuda.mem_get_info()[0]
    return torch.empty(free - (mb << 20), dtype=torch.uint8, device="cuda")
"""

# two state blocks of 67 MB fit, the four of the sweep do not
SQUARE = """
lat = capi.tbpm_lattice_create(ctx, capi.lattice_desc(0, (2048, 1024), t=1.0, W=1.0, seed=3))
req = S(n_states=4, n_moments=64, state_seed=5)
kept = fill(215)
mu = np.zeros((4, 64, 2)); capi.tbpm_moments(ctx, lat, req, mu)
del kept; torch.cuda.empty_cache()
ref = np.zeros_like(mu); capi.tbpm_moments(ctx, lat, req, ref)
assert np.max(np.abs(mu - ref)) <= 1e-6
"""

# a quarter of the sites vacant: two compact blocks of 25 MB fit, four of 34 MB do not
VACANCY = """
lat = capi.tbpm_lattice_create(ctx, capi.lattice_desc(1, (1024, 1024), t=-2.7, W=1.0, seed=3, vacancy_frac=0.25))
req = S(n_states=2, n_moments=64, state_seed=5)
kept = fill(100)
mu = np.zeros((2, 64, 2)); capi.tbpm_moments(ctx, lat, req, mu)
del kept; torch.cuda.empty_cache()
ref = np.zeros_like(mu); capi.tbpm_moments(ctx, lat, req, ref)
assert np.max(np.abs(mu - ref)) <= 1e-6
"""

# per-CTA sums of 50,000 resident steps take 384 MB; the one-step pass needs none of it
RESIDENT = """
lat = capi.tbpm_lattice_create(ctx, capi.lattice_desc(0, (60, 60), t=1.0, W=1.0, seed=3))
req = S(n_states=8, n_moments=100000, state_seed=5)
kept = fill(150)
mu = np.zeros((8, 100000, 2)); capi.tbpm_moments(ctx, lat, req, mu)
del kept; torch.cuda.empty_cache()
ref = np.zeros_like(mu); capi.tbpm_moments(ctx, lat, req, ref)
assert np.max(np.abs(mu - ref)) <= 1e-4
"""

# 16 kets and the propagation fit on the 55 % of the sites that are there, not on all of them
CONDUCTIVITY = """
lat = capi.tbpm_lattice_create(ctx, capi.lattice_desc(1, (1024, 1024), t=-2.7, W=1.0, seed=3, vacancy_frac=0.45))
E = np.linspace(-4.0, 4.0, 16)
req = S(n_states=1, form=2, n_steps=6, time_block=2, state_seed=5)
C, sg = np.zeros((1, 16, 7), np.complex128), np.zeros((1, 16))
kept = fill(340)
capi.tbpm_conductivity(ctx, lat, req, 0, E, C, sg)
del kept; torch.cuda.empty_cache()
C2, sg2 = np.zeros_like(C), np.zeros_like(sg)
capi.tbpm_conductivity(ctx, lat, req, 0, E, C2, sg2)
assert np.max(np.abs(C - C2)) <= 3e-5 * np.max(np.abs(C2))
"""

# windows of the first call limited by memory: the second call gets the same ones
REPEATED = """
lat = capi.tbpm_lattice_create(ctx, capi.lattice_desc(1, (1024, 1024), t=-2.7, W=1.0, seed=3))
req = S(n_states=1, form=2, n_steps=8, time_block=4, state_seed=5)
opt = S(n_states=1, form=2, n_steps=4, time_block=2, state_seed=5)
kept = fill(700)
for call in (lambda o: capi.tbpm_correlation(ctx, lat, req, o[0]),
             lambda o: capi.tbpm_optical_conductivity(ctx, lat, opt, 0, 0, 0.1, 0.5, 4.0, 8, o[1], o[2])):
    runs = []
    for k in range(3):
        out = [np.zeros((1, 9), np.complex128), np.zeros((1, 5), np.complex128), np.zeros((1, 8), np.complex128)]
        n = capi.tbpm_launch_count(ctx); call(out)
        runs.append((capi.tbpm_launch_count(ctx) - n, out))
    for n, out in runs[1:]:
        assert n == runs[0][0], [r[0] for r in runs]
        assert all(np.array_equal(a, b) for a, b in zip(out, runs[0][1]))
"""

CASES = dict(square=SQUARE, vacancy=VACANCY, resident=RESIDENT, conductivity=CONDUCTIVITY, repeated=REPEATED)


@pytest.mark.parametrize("name", CASES)
def test_little_memory(name):
    r = subprocess.run([sys.executable, "-c", PRELUDE.format(root=ROOT) + CASES[name]], capture_output=True, text=True,
                       timeout=600, cwd=ROOT)
    assert r.returncode == 0, r.stdout[-1000:] + r.stderr[-3000:]
