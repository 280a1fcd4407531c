"""Every synchronous call reports a bounded wait that expired in its kernels.

The register sweep, its window passes and the resident recurrence record an expired wait in the
context's status word and return; results formed after that are void.  Here the word is written
from the host (no wait expires on the device): each call must return TBPM_ETIMEOUT once, and the
same call made again must succeed.  A cooperative launch that the driver refuses is no failure either."""
import ctypes as C
import os
import shutil
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def capi():
    import __graft_entry__
    __graft_entry__.build()
    from paper_2510_17432_gb300 import capi as c
    return c


@pytest.fixture(scope="module")
def poke(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    out = str(tmp_path_factory.mktemp("status") / "libstatus_word.so")
    subprocess.run([nvcc, "-std=c++17", "-shared", "-Xcompiler", "-fPIC", "-gencode", "arch=compute_103a,code=sm_103a",
                    "-I", os.path.join(ROOT, "include"), "-I", os.path.join(ROOT, "paper_2510_17432_gb300", "csrc"),
                    "-o", out, os.path.join(ROOT, "tests", "status_word.cu")], check=True, capture_output=True)
    lib = C.CDLL(out)
    lib.set_status_word.argtypes = [C.c_void_p, C.c_int]
    lib.set_num_sms.argtypes = [C.c_void_p, C.c_int]
    return lib


S, NT, NE = 2, 4, 3


def _calls(capi, ctx, lat, n):
    E = np.array([-0.5, 0.1, 0.6])
    q = lambda **kw: capi.request(n_states=S, state_seed=3, **kw)  # noqa: E731
    Cc, Cw = np.zeros((S, NT + 1), np.complex128), np.zeros((S, NE, NT + 1), np.complex128)
    block = q(form=2, n_steps=NT, time_block=2)
    return {
        "moments": lambda: capi.tbpm_moments(ctx, lat, q(n_moments=16), np.zeros((S, 16, 2))),
        "dos": lambda: capi.tbpm_dos(ctx, lat, q(n_moments=16), E, np.zeros((S, NE))),
        "correlation": lambda: capi.tbpm_correlation(ctx, lat, block, Cc),
        "correlation_moment_form": lambda: capi.tbpm_correlation(ctx, lat, q(form=1, n_steps=NT), Cc),
        "quasi_eigenstates": lambda: capi.tbpm_quasi_eigenstates(ctx, lat, q(form=3, n_steps=NT), E,
                                                                 np.zeros((NE, S, n), np.complex64)),
        "conductivity": lambda: capi.tbpm_conductivity(ctx, lat, block, 0, E, Cw, np.zeros((S, NE))),
        "fermi_apply": lambda: capi.tbpm_fermi_apply(ctx, lat, q(), 0.1, 0.5, False, np.zeros((S, n), np.complex64)),
        "optical_conductivity": lambda: capi.tbpm_optical_conductivity(ctx, lat, block, 0, 0, 0.1, 0.5, 4.0, 8, Cc,
                                                                       np.zeros((S, 8), np.complex128)),
        "polarization": lambda: capi.tbpm_polarization(ctx, lat, block, (0.1, 0.0, 0.0), 0.1, 0.5, E, Cc,
                                                       np.zeros((S, NE), np.complex128)),
        "charge_density": lambda: capi.tbpm_charge_density(ctx, lat, block, 0.1, 0.5, np.zeros((S, n))),
        "block_autotune": lambda: capi.tbpm_block_autotune(ctx, lat, block, NT),
        "sync": lambda: capi.tbpm_sync(ctx),
    }


def test_synchronous_calls_report_an_expired_wait_once(capi, poke):
    ctx = capi.tbpm_create(0)
    try:
        lat = capi.tbpm_lattice_create(ctx, capi.lattice_desc(1, (130, 40), t=-2.7, W=1.0, seed=3))
        missed = []
        for name, call in _calls(capi, ctx, lat, capi.tbpm_lattice_info(lat).n_sites).items():
            call()
            poke.set_status_word(ctx, 1)
            try:
                call()
                missed.append(name)
                poke.set_status_word(ctx, 0)
            except capi.TbpmError as e:
                assert e.status == -4, (name, str(e))
            call()
        assert not missed
        capi.tbpm_lattice_destroy(lat)
    finally:
        capi.tbpm_destroy(ctx)


def test_a_cooperative_grid_that_does_not_fit_takes_another_pass(capi, poke):
    """A context that believes in more SMs than there are plans 256 CTAs of 205 KB, one to an SM; the launch is
    refused on the host and the request runs in the register sweep."""
    mu = []
    for sms in (0, 300):
        ctx = capi.tbpm_create(0)
        try:
            lat = capi.tbpm_lattice_create(ctx, capi.lattice_desc(0, (360, 1024), t=1.0, W=1.0, seed=3))
            if sms:
                poke.set_num_sms(ctx, sms)
            mu.append(np.zeros((8, 32, 2)))
            capi.tbpm_moments(ctx, lat, capi.request(n_states=8, n_moments=32, state_seed=3), mu[-1])
            capi.tbpm_lattice_destroy(lat)
        finally:
            capi.tbpm_destroy(ctx)
    assert np.max(np.abs(mu[0] - mu[1])) <= 1e-6
