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


@pytest.mark.parametrize("L,S", [((64, 32), 32), ((1024, 1024), 8)])
def test_random_phases_are_the_fp64_ones(capi, ctx, L, S):
    """FP32 states are the FP64 ones rounded, ties and all: the FP32 evaluation alone missed one value in 400,000."""
    lat = capi.tbpm_lattice_create(ctx, capi.lattice_desc(capi.HONEYCOMB, L, t=1.0))
    n = capi.tbpm_lattice_info(lat).n_sites
    a, b = np.zeros((S, n), np.complex64), np.zeros((S, n), np.complex128)
    capi.tbpm_states_export(ctx, lat, capi.request(n_states=S, state_seed=12), a)
    capi.tbpm_states_export(ctx, lat, capi.request(n_states=S, state_seed=12, precision=1), b)
    capi.tbpm_lattice_destroy(lat)
    assert np.array_equal(a, b.astype(np.complex64))


def _pair(capi, ctx, spec):
    lat = capi.tbpm_lattice_create(ctx, capi.lattice_desc(spec["kind"], spec["L"], t=spec["t"], W=spec["W"], seed=77,
                                                          vacancy_frac=spec.get("vac", 0.0),
                                                          pbc=spec.get("pbc", (1, 1, 1))))
    ol = olat.build_lattice(spec["kind"], (tuple(spec["L"]) + (1,))[:3], t=spec["t"], W=spec["W"], seed=77,
                            vacancy_frac=spec.get("vac", 0.0), pbc=spec.get("pbc", (1, 1, 1)))
    return lat, ol


# Shapes of the register sweep beyond honeycomb pairs: the square lattice (even and odd rows, so that
# the last cell holds one or two sites; one band and several; open and periodic), one state per site
# (128-cell bands), and vacancy lattices in the full layout.  M / 2 = 4 k + 1 .. 4 k + 4 steps: every
# tail of the last pass.
SWEEPS = [
    ("square_one_band", dict(kind=0, L=(128, 96), t=1.0, W=0.0), 4, 42),
    ("square_odd_W", dict(kind=0, L=(131, 97), t=1.0, W=1.0), 8, 44),
    ("square_odd_open_x", dict(kind=0, L=(197, 99), t=-1.0, W=0.7, pbc=(0, 1, 1)), 5, 46),
    ("square_open_y_S32", dict(kind=0, L=(96, 101), t=1.0, W=2.0, pbc=(1, 0, 1)), 32, 40),
    ("square_open_xy_S2", dict(kind=0, L=(301, 120), t=1.0, W=0.0, pbc=(0, 0, 1)), 2, 42),
    ("square_S1", dict(kind=0, L=(258, 98), t=1.0, W=1.0), 1, 46),
    ("square_S1_open", dict(kind=0, L=(512, 100), t=1.0, W=0.0, pbc=(0, 0, 1)), 1, 40),
    ("honey_S1", dict(kind=1, L=(128, 32), t=-2.7, W=0.0), 1, 44),
    ("honey_S1_W_open", dict(kind=1, L=(253, 51), t=-2.7, W=1.0, pbc=(0, 0, 1)), 1, 42),
    ("honey_vac_S1", dict(kind=1, L=(150, 61), t=-2.7, W=1.0, vac=0.03), 1, 46),
    ("honey_vac_clean_S3", dict(kind=1, L=(64, 40), t=-2.7, W=0.0, vac=0.2, pbc=(1, 0, 1)), 3, 40),
    ("honey_vac_open_x_S8", dict(kind=1, L=(70, 45), t=1.0, W=0.5, vac=0.4, pbc=(0, 1, 1)), 8, 42),
    ("square_vac_S2", dict(kind=0, L=(257, 99), t=1.0, W=1.0, vac=0.05), 2, 44),
    ("square_vac_S1", dict(kind=0, L=(256, 97), t=1.0, W=0.3, vac=0.1), 1, 46),
]


def _moments(capi, ctx, lat, S, M, mode, sites=None):
    mu = np.zeros((S, M, 2))
    capi.tbpm_set_fusion(ctx, mode)
    try:
        capi.tbpm_moments(ctx, lat, capi.request(n_states=S, n_moments=M, state_seed=3, sites=sites), mu)
    finally:
        capi.tbpm_set_fusion(ctx, 8)
    return mu[..., 0] + 1j * mu[..., 1]


@pytest.mark.parametrize("name,spec,S,M", SWEEPS, ids=[c[0] for c in SWEEPS])
def test_sweep_shapes_match_the_one_step_pass_and_the_oracle(capi, ctx, name, spec, S, M):
    lat, ol = _pair(capi, ctx, spec)
    capi.tbpm_set_fusion(ctx, 8)
    assert capi.tbpm_moment_pass_kind(ctx, lat, capi.request(n_states=S, n_moments=M)) == capi.PASS_SWEEP
    got, one = _moments(capi, ctx, lat, S, M, 8), _moments(capi, ctx, lat, S, M, 0)
    assert np.max(np.abs(got - one)) <= 1e-6
    psi = oprop.random_phase_states(ol, 3, S)
    for s in {0, S - 1}:
        assert np.max(np.abs(got[s] - oprop.moments(ol, psi[s], psi[s], M))) <= 1e-5
    sites = np.array([0, ol.n - 1, ol.n // 2], np.int64)  # site states: no averaging over the lattice
    got = _moments(capi, ctx, lat, 3, M, 8, sites)
    for k, i in enumerate(sites):
        e = np.zeros(ol.n, np.complex128)
        e[i] = 1.0
        assert np.max(np.abs(got[k] - oprop.moments(ol, e, e, M))) <= 1e-5
    capi.tbpm_lattice_destroy(lat)


# Vacancy honeycombs narrower than the bands of modes 9 and 10 (192 / P and 256 / P cells) and not than the
# masked sweep's own (128 / P): the masked sweep has 128 threads in every mode.
NARROW = [
    ("S2_below_192", dict(kind=1, L=(190, 33), t=-2.7, W=1.0, vac=0.01), 2),
    ("S2_below_256", dict(kind=1, L=(200, 40), t=-2.7, W=0.0, vac=0.05), 2),
    ("S4_one_band", dict(kind=1, L=(64, 37), t=-2.7, W=0.5, vac=0.1, pbc=(1, 0, 1)), 4),
    ("S8_between", dict(kind=1, L=(50, 32), t=1.0, W=0.0, vac=0.02, pbc=(0, 1, 1)), 8),
]


@pytest.mark.parametrize("mode", [8, 9, 10])
@pytest.mark.parametrize("name,spec,S", NARROW, ids=[c[0] for c in NARROW])
def test_wide_modes_on_narrow_vacancy_lattices(capi, ctx, name, spec, S, mode):
    lat, ol = _pair(capi, ctx, spec)
    M = 42
    got = _moments(capi, ctx, lat, S, M, mode)
    psi = oprop.random_phase_states(ol, 3, S)
    for s in {0, S - 1}:
        assert np.max(np.abs(got[s] - oprop.moments(ol, psi[s], psi[s], M))) <= 1e-5
    capi.tbpm_lattice_destroy(lat)


WINDOWS = [
    ("square", dict(kind=0, L=(129, 97), t=1.0, W=1.0, pbc=(1, 0, 1)), 4),
    ("square_S1", dict(kind=0, L=(256, 96), t=1.0, W=1.0), 1),
    ("honey_S1", dict(kind=1, L=(130, 40), t=-2.7, W=1.0), 1),
    ("honey_vac_S1", dict(kind=1, L=(140, 40), t=-2.7, W=1.0, vac=0.05), 1),
    ("honey_vac_S2", dict(kind=1, L=(130, 33), t=-2.7, W=0.0, vac=0.1), 2),
]


@pytest.mark.parametrize("name,spec,S", WINDOWS, ids=[c[0] for c in WINDOWS])
def test_window_passes_of_the_new_shapes(capi, ctx, name, spec, S):
    """Correlations in every form, quasi-eigenstates and the conductivity through the window passes."""
    from oracle import conductivity as oec, quasi as oqe
    lat, ol = _pair(capi, ctx, spec)
    psi = oprop.random_phase_states(ol, 8, S)
    s = S - 1
    Nt = 19
    ref = oprop.correlation_sequential(ol, psi[s], Nt, np.pi)
    for form, b in ((0, 0), (2, 5), (2, 0)):
        C = np.zeros((S, Nt + 1), np.complex128)
        capi.tbpm_correlation(ctx, lat, capi.request(n_states=S, form=form, n_steps=Nt, time_block=b, state_seed=8), C)
        assert np.max(np.abs(C[s] - ref)) <= 1e-5, form
    E = ol.H0 + np.array([-0.6, 0.05, 0.4]) * (ol.E_max - ol.E_min) / 2
    out = np.zeros((E.size, S, ol.n), np.complex64)
    qref = oqe.qe_concurrent_e(ol, psi[s], E, Nt)
    for form in (3, 2):
        capi.tbpm_quasi_eigenstates(ctx, lat, capi.request(n_states=S, form=form, n_steps=Nt, state_seed=8), E, out)
        for k in range(E.size):
            assert np.max(np.abs(out[k, s] - qref[k])) <= 1e-5 * np.max(np.abs(qref[k])), (form, k)
    for form in (0, 1, 2):
        C = np.zeros((S, E.size, Nt + 1), np.complex128)
        sigma = np.zeros((S, E.size))
        capi.tbpm_conductivity(ctx, lat, capi.request(n_states=S, form=form, n_steps=Nt, state_seed=8), 0, E, C, sigma)
        Cref, _ = oec.ec_correlation_sequential(ol, psi[s], E, Nt, 0)
        for k in range(E.size):
            assert np.max(np.abs(C[s, k] - Cref[k])) <= 3e-5 * np.max(np.abs(Cref[k])), (form, k)
    capi.tbpm_lattice_destroy(lat)


# Small lattices whose whole recurrence runs in one launch: one line per CTA and several, fewer lines than
# CTAs, a ragged last CTA, a lattice near the shared-memory limit, every kind and boundary, widths of one
# and two cells, both precisions, and M / 2 around the batches of eight steps whose sums are stored together.
RESIDENT = [
    ("square64_c128", dict(kind=0, L=(64, 64), t=1.0, W=1.0), 1, 1, 96),
    ("square_thin_c128", dict(kind=0, L=(2, 300), t=1.0, W=0.5), 3, 1, 34),
    ("square_one_row", dict(kind=0, L=(50, 1), t=1.0, W=1.0), 2, 0, 32),
    ("honey_ribbon", dict(kind=1, L=(45, 47), t=1.0, W=1.0, pbc=(1, 0, 1)), 4, 0, 48),
    ("honey_two_cells_open", dict(kind=1, L=(2, 155), t=-2.7, W=0.0, pbc=(0, 1, 1)), 1, 0, 50),
    ("honey_c128_S5", dict(kind=1, L=(31, 160), t=-2.7, W=1.0), 5, 1, 30),
    ("cubic_S32", dict(kind=2, L=(7, 9, 11), t=1.0, W=1.5, pbc=(1, 1, 0)), 32, 0, 20),
    ("cubic_c128", dict(kind=2, L=(12, 5, 8), t=1.0, W=0.3, pbc=(0, 1, 1)), 2, 1, 18),
    ("cubic_lines_over_ctas", dict(kind=2, L=(10, 31, 13), t=1.0, W=2.0), 8, 0, 16),
    ("square_large_S2", dict(kind=0, L=(95, 2900), t=1.0, W=0.0), 2, 0, 12),
    ("square_large_S1", dict(kind=0, L=(61, 9000), t=1.0, W=1.0, pbc=(1, 0, 1)), 1, 0, 36),
]


@pytest.mark.parametrize("name,spec,S,prec,M", RESIDENT, ids=[c[0] for c in RESIDENT])
def test_resident_recurrence_matches_the_oracle(capi, name, spec, S, prec, M):
    ctx = capi.tbpm_create(0)  # the resident kernel is the default; a chosen mode may name another pass
    try:
        lat, ol = _pair(capi, ctx, spec)
        req = capi.request(n_states=S, precision=prec, n_moments=M, state_seed=3)
        mu = np.zeros((S, M, 2))
        capi.tbpm_moments(ctx, lat, req, mu)
        again = np.zeros_like(mu)
        launches = capi.tbpm_launch_count(ctx)
        capi.tbpm_moments(ctx, lat, req, again)
        assert capi.tbpm_launch_count(ctx) - launches == 3  # states, recurrence, sums
        assert np.array_equal(mu, again)
        capi.tbpm_set_fusion(ctx, 0)
        one = np.zeros_like(mu)
        capi.tbpm_moments(ctx, lat, req, one)
        assert np.max(np.abs(mu - one)) <= (1e-12 if prec else 1e-6)
        psi = oprop.random_phase_states(ol, 3, S)
        for s in {0, S - 1}:
            ref = oprop.moments(ol, psi[s], psi[s], M)
            assert np.max(np.abs(mu[s, :, 0] + 1j * mu[s, :, 1] - ref)) <= (1e-11 if prec else 1e-5)
        capi.tbpm_lattice_destroy(lat)
    finally:
        capi.tbpm_destroy(ctx)


def test_the_reported_pass_is_the_one_that_runs(capi):
    """By default, under each mode set (the documented default 8 as well), and with the default brought back: the
    reported kind, and the launches of the request (resident: states, recurrence, sums; else one a pass or step)."""
    M = 64
    cases = [  # lattice, states, precision; kinds by default, in mode 8, in mode 0
        (dict(kind=1, L=(100, 64), t=-2.7, W=1.0), 4, 0, "RESIDENT", "SWEEP", "STENCIL"),
        (dict(kind=1, L=(100, 64), t=-2.7, W=1.0), 1, 0, "RESIDENT", "STENCIL", "STENCIL"),
        (dict(kind=1, L=(200, 180), t=-2.7, W=1.0), 4, 0, "SWEEP", "SWEEP", "STENCIL"),
        (dict(kind=0, L=(64, 64), t=1.0, W=1.0), 1, 1, "RESIDENT", "STENCIL", "STENCIL"),
        (dict(kind=0, L=(128, 96), t=1.0, W=1.0), 4, 0, "RESIDENT", "SWEEP", "STENCIL"),
        (dict(kind=2, L=(9, 8, 7), t=1.0, W=1.0), 2, 0, "RESIDENT", "STENCIL", "STENCIL"),
    ]
    launches = {"RESIDENT": 3, "SWEEP": 1 + M // 8, "STENCIL": 1 + M // 2}
    ctx = capi.tbpm_create(0)
    try:
        capi.tbpm_set_graphs(ctx, False)
        for spec, S, prec, *kinds in cases:
            lat = capi.tbpm_lattice_create(ctx, capi.lattice_desc(seed=3, **spec))
            req = capi.request(n_states=S, precision=prec, n_moments=M, state_seed=3)
            for mode, want in zip((None, 8, 0, None), kinds + [kinds[0]]):
                if mode is None:  # the default, by the call that brings it back
                    capi.tbpm_set_fusion(ctx, 8)
                    capi.tbpm_set_resident(ctx, True)
                else:
                    capi.tbpm_set_fusion(ctx, mode)
                assert capi.tbpm_moment_pass_kind(ctx, lat, req) == getattr(capi, "PASS_" + want), (spec, mode)
                mu = np.zeros((S, M, 2))
                capi.tbpm_moments(ctx, lat, req, mu)
                n = capi.tbpm_launch_count(ctx)
                capi.tbpm_moments(ctx, lat, req, mu)
                assert capi.tbpm_launch_count(ctx) - n == launches[want], (spec, mode, want)
            capi.tbpm_lattice_destroy(lat)
    finally:
        capi.tbpm_destroy(ctx)
    ctx = capi.tbpm_create(0)  # and without any call
    try:
        lat = capi.tbpm_lattice_create(ctx, capi.lattice_desc(1, (100, 64), t=-2.7, W=1.0, seed=3))
        assert capi.tbpm_moment_pass_kind(ctx, lat, capi.request(n_states=4, n_moments=M)) == capi.PASS_RESIDENT
        capi.tbpm_lattice_destroy(lat)
    finally:
        capi.tbpm_destroy(ctx)


# The cubic march: tiles cut at every edge, lattices of one tile and less, one and two planes, every number of
# state pairs per CTA, segments of planes, open boundaries, both precisions.
MARCH = [
    ("tile_and_one_S8", (9, 9, 5), dict(), 8, 0),
    ("one_plane_S1", (33, 7, 1), dict(), 1, 0),
    ("two_planes_open_z", (5, 4, 2), dict(pbc=(1, 1, 0)), 2, 0),
    ("thin_x_S32", (1, 17, 6), dict(), 32, 0),
    ("open_all_S16", (13, 21, 9), dict(pbc=(0, 0, 0)), 16, 0),
    ("many_segments_S4", (8, 8, 200), dict(), 4, 0),
    ("c128_S3", (10, 11, 12), dict(pbc=(0, 1, 1)), 3, 1),
    ("c128_S1_wide", (70, 3, 4), dict(pbc=(1, 0, 1)), 1, 1),
]


@pytest.mark.parametrize("name,L,kw,S,prec", MARCH, ids=[c[0] for c in MARCH])
def test_cubic_march_matches_the_oracle(capi, ctx, name, L, kw, S, prec):
    spec = dict(kind=2, L=L, t=1.0, W=1.0, **kw)
    lat, ol = _pair(capi, ctx, spec)
    psi = oprop.random_phase_states(ol, 3, S)
    M, Nt = 18, 7
    mu = np.zeros((S, M, 2))
    capi.tbpm_set_fusion(ctx, 0)  # one step per launch
    try:
        capi.tbpm_moments(ctx, lat, capi.request(n_states=S, precision=prec, n_moments=M, state_seed=3), mu)
    finally:
        capi.tbpm_set_fusion(ctx, 8)
    C = np.zeros((S, Nt + 1), np.complex128)
    capi.tbpm_correlation(ctx, lat, capi.request(n_states=S, precision=prec, form=2, n_steps=Nt, time_block=4,
                                                 state_seed=3), C)
    tol = 1e-11 if prec else 1e-5
    for s in {0, S - 1}:
        assert np.max(np.abs(mu[s, :, 0] + 1j * mu[s, :, 1] - oprop.moments(ol, psi[s], psi[s], M))) <= tol
        assert np.max(np.abs(C[s] - oprop.correlation_sequential(ol, psi[s], Nt, np.pi))) <= tol
    capi.tbpm_lattice_destroy(lat)


# The tap kernel: rows of an odd number of sites (cells of two), tiles cut by one and short by one, open and
# wrapped halos, a lattice smaller than the halo, and the longest hopping there is.
TAPS = [
    ("odd_periodic", (129, 33), dict(kind=0, cutoff=3.3), 2),
    ("odd_open_x", (127, 31), dict(kind=0, cutoff=2.1, pbc=(0, 1, 1)), 3),
    ("one_column", (1, 40), dict(kind=0, cutoff=2.1), 2),
    ("nearest_only_open", (5, 7), dict(kind=0, cutoff=1.0, pbc=(0, 0, 1)), 4),
    ("honeycomb_cells", (65, 33), dict(kind=1, cutoff=5.1, pbc=(1, 0, 1)), 2),
    ("honeycomb_images", (3, 2), dict(kind=1, cutoff=5.1), 2),
    ("longest_square", (131, 37), dict(kind=0, cutoff=12.0), 2),
    ("longest_honeycomb", (67, 30), dict(kind=1, cutoff=12.0), 3),
]


@pytest.mark.parametrize("name,L,kw,S", TAPS, ids=[c[0] for c in TAPS])
def test_tap_kernel_matches_the_oracle(capi, ctx, name, L, kw, S):
    kind, pbc, cutoff = kw["kind"], kw.get("pbc", (1, 1, 1)), kw["cutoff"]
    lat = capi.tbpm_lattice_create(ctx, capi.lattice_desc(kind, L, t=1.0, W=0.5, seed=7, pbc=pbc, cutoff=cutoff,
                                                          decay=0.6))
    ol = olat.build_lattice(kind, L + (1,), t=1.0, W=0.5, seed=7, pbc=pbc, cutoff=cutoff, decay=0.6)
    M = 18
    mu = np.zeros((S, M, 2))
    capi.tbpm_moments(ctx, lat, capi.request(n_states=S, n_moments=M, state_seed=3), mu)
    psi = oprop.random_phase_states(ol, 3, S)
    for s in {0, S - 1}:
        assert np.max(np.abs(mu[s, :, 0] + 1j * mu[s, :, 1] - oprop.moments(ol, psi[s], psi[s], M))) <= 1e-5
    capi.tbpm_lattice_destroy(lat)
