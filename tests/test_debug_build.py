"""The index-checked debug build (TBPM_DEBUG): the hot kernels skip and record out-of-range
global indices instead of trapping, and tbpm_debug_status() reports the first one per unit.

Without a GPU: the debug library builds and exports the status call, the regular library
answers TBPM_EUNSUPPORTED with zero words, and the status words decode.  With a GPU: every
kernel family that carries checks runs on valid inputs through the debug library with all
words clean, and its moments equal the regular library's bit for bit (the checks change no
arithmetic)."""
import ctypes as C

import numpy as np
import pytest


@pytest.fixture(scope="module")
def capi():
    import __graft_entry__
    __graft_entry__.build()
    from paper_2510_17432_gb300 import _build, capi as c
    _build.build(debug=True)
    return c


def test_debug_library_exports_the_status_call(capi):
    lib = capi.load_debug()
    assert hasattr(lib, "tbpm_debug_status") and hasattr(lib, "tbpm_moments")


def test_regular_library_reports_unsupported(capi):
    # no device work: the regular build answers before touching CUDA; a context handle is not
    # needed for that answer, but NULL is rejected first, so pass a dummy pointer
    words = (C.c_uint64 * 3)(7, 7, 7)
    st = capi.load().tbpm_debug_status(C.c_void_p(1), words)
    assert st == -5 and list(words) == [0, 0, 0]
    assert capi.load().tbpm_debug_status(None, words) == -1


def test_status_words_decode(capi):
    assert capi.decode_debug_word(0) is None
    assert capi.decode_debug_word((3 << 48) | 12345) == ("sweep store", 12345)
    assert capi.decode_debug_word((2 << 48) | 0xFFFFFFFFFFFF) == ("ELL neighbour index", 0xFFFFFFFFFFFF)


@pytest.mark.gpu
def test_checked_kernels_stay_clean_and_exact(capi):
    dbg = capi.load_debug()
    cases = [  # (lattice, states, moments): register sweep, stencil, ELL, serving-sized stencil
        (dict(kind=1, L=(100, 64), t=-2.7, W=1.0, seed=3), 8, 256),
        (dict(kind=0, L=(64, 48), t=1.0, W=1.0, seed=3), 4, 128),
        (dict(kind=1, L=(40, 30), t=-2.7, W=1.0, vacancy_frac=0.05, seed=3), 2, 128),
        (dict(kind=2, L=(12, 10, 9), t=1.0, W=0.5, seed=3), 1, 64),
    ]
    results = {}
    for name, lib in (("debug", dbg), ("regular", capi.load())):
        h = C.c_void_p()
        assert lib.tbpm_create(C.byref(h), 0) == 0
        try:
            for k, (ld, S, M) in enumerate(cases):
                lat = C.c_void_p()
                assert lib.tbpm_lattice_create(h, C.byref(capi.lattice_desc(**ld)), C.byref(lat)) == 0
                mu = np.zeros((S, M, 2))
                req = capi.request(n_states=S, precision=0, n_moments=M, state_seed=5)
                assert lib.tbpm_moments(h, lat, C.byref(req), mu.ctypes.data_as(C.c_void_p)) == 0
                results[(name, k)] = mu
                lib.tbpm_lattice_destroy(lat)
            if name == "debug":
                words = capi.tbpm_debug_status(h, lib)
                assert words == [0, 0, 0], [capi.decode_debug_word(w) for w in words]
        finally:
            lib.tbpm_destroy(h)
    for k in range(len(cases)):
        assert np.array_equal(results[("debug", k)], results[("regular", k)])


def test_status_words_of_the_newer_kernels_decode(capi):
    for kid, name in ((6, "resident units"), (7, "cubic march units"), (8, "flush units"), (9, "tap kernel units")):
        assert capi.decode_debug_word((kid << 48) | 7) == (name, 7)


@pytest.mark.gpu
def test_every_checked_kernel_is_reached_and_stays_clean(capi):
    """Each kernel with checks by its own route (the reported pass, or a correlation through window and flush) on
    sizes that are no multiple of its tiles: words clean, results equal to the regular library's bit for bit."""
    dbg = capi.load_debug()
    SWEEP, STENCIL, ELL, RES, TAPS = (capi.PASS_SWEEP, capi.PASS_STENCIL, capi.PASS_ELL, capi.PASS_RESIDENT,
                                      capi.PASS_TAPS)
    honey, square, cubic = dict(kind=1, t=-2.7, seed=3), dict(kind=0, t=1.0, seed=3), dict(kind=2, t=1.0, seed=3)
    cases = [  # lattice, states, precision, fusion mode (None: default), expected pass
        (dict(honey, L=(100, 64), W=1.0), 8, 0, 8, SWEEP),
        (dict(honey, L=(131, 33), W=1.0, pbc=(1, 0, 1)), 1, 0, 8, SWEEP),
        (dict(honey, L=(100, 47), W=0.0, vacancy_frac=0.1), 4, 0, 8, SWEEP),
        (dict(square, L=(131, 97), W=1.0, pbc=(0, 1, 1)), 4, 0, 8, SWEEP),
        (dict(square, L=(64, 48), W=1.0), 4, 0, 0, STENCIL),
        (dict(cubic, L=(13, 9, 11), W=1.0, pbc=(1, 0, 1)), 8, 0, 0, STENCIL),  # the march
        (dict(cubic, L=(1, 17, 6), W=0.5), 3, 1, 0, STENCIL),
        (dict(honey, L=(45, 47), W=1.0, pbc=(1, 0, 1)), 4, 0, None, RES),
        (dict(square, L=(50, 170), W=1.0), 2, 1, None, RES),
        (dict(cubic, L=(7, 9, 11), W=0.0), 32, 0, None, RES),
        (dict(honey, L=(40, 30), W=1.0, vacancy_frac=0.05), 2, 0, None, ELL),
        (dict(square, L=(129, 33), W=0.5, cutoff=3.3, decay=0.6), 3, 0, None, TAPS),
        (dict(honey, L=(65, 33), W=0.0, cutoff=5.1, decay=0.6, pbc=(1, 0, 1)), 2, 0, None, TAPS),
    ]
    M, NT = 50, 9
    results = {}
    for name, lib in (("debug", dbg), ("regular", capi.load())):
        for k, (ld, S, prec, mode, want) in enumerate(cases):
            h, lat, kind = C.c_void_p(), C.c_void_p(), C.c_int(-1)
            assert lib.tbpm_create(C.byref(h), 0) == 0
            try:
                if mode is not None:
                    assert lib.tbpm_set_fusion(h, mode) == 0
                assert lib.tbpm_lattice_create(h, C.byref(capi.lattice_desc(**ld)), C.byref(lat)) == 0
                req = capi.request(n_states=S, precision=prec, n_moments=M, state_seed=5)
                assert lib.tbpm_moment_pass_kind(h, lat, C.byref(req), C.byref(kind)) == 0 and kind.value == want, k
                mu, corr = np.zeros((S, M, 2)), np.zeros((S, NT + 1), np.complex128)
                assert lib.tbpm_moments(h, lat, C.byref(req), mu.ctypes.data_as(C.c_void_p)) == 0
                req = capi.request(n_states=S, precision=prec, form=2, n_steps=NT, time_block=5, state_seed=5)
                assert lib.tbpm_correlation(h, lat, C.byref(req), corr.ctypes.data_as(C.c_void_p)) == 0
                results[(name, k)] = (mu, corr)
                lib.tbpm_lattice_destroy(lat)
                if name == "debug":
                    words = capi.tbpm_debug_status(h, lib)
                    assert words == [0, 0, 0], (k, [capi.decode_debug_word(w) for w in words])
            finally:
                lib.tbpm_destroy(h)
    for k in range(len(cases)):
        for a, b in zip(results[("debug", k)], results[("regular", k)]):
            assert np.isfinite(a).all() and np.array_equal(a, b), k
