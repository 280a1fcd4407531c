"""Edges of the kernels' own ranges: the random-phase evaluation, and the sizes around tiles, bands
and remainders of the fused passes, against the FP64 oracle."""
import numpy as np
import pytest

from oracle import lattice as olat, propagate as oprop

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def capi():
    import __graft_entry__
    __graft_entry__.build()
    from paper_2510_17432_gb300 import capi as c
    return c


@pytest.fixture(scope="module")
def ctx(capi):
    h = capi.tbpm_create(0)
    yield h
    capi.tbpm_destroy(h)


@pytest.mark.parametrize("L,S", [((1, 1), 1), ((37, 29), 3), ((300, 211), 2)])
def test_random_phases_are_rounded_once(capi, ctx, L, S):
    """The FP32 phases differ from the FP64 ones rounded to FP32 by at most one ulp, and only near ties
    (the evaluation's own error is below 2^-10 ulp: fewer than one value in a thousand may differ)."""
    desc = capi.lattice_desc(capi.HONEYCOMB, L, t=1.0)
    lat = capi.tbpm_lattice_create(ctx, desc)
    n = capi.tbpm_lattice_info(lat).n_sites
    out = np.zeros((S, n), np.complex64)
    capi.tbpm_states_export(ctx, lat, capi.request(n_states=S, state_seed=11), out)
    capi.tbpm_lattice_destroy(lat)
    ol = olat.build_lattice(1, L + (1,), t=1.0, W=0.0, seed=1)
    want = np.asarray(oprop.random_phase_states(ol, 11, S)).astype(np.complex64)
    a, b = out.view(np.float32).ravel(), want.view(np.float32).ravel()
    assert np.all(np.abs(a - b) <= np.spacing(np.abs(b)))
    assert np.count_nonzero(a != b) <= a.size // 1000
