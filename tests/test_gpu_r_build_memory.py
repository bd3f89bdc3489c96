"""Region building where device memory is short: without room for the beam, and
with the beam given back half-way, the results are those with it, bit for bit."""
import numpy as np
import pytest

from paper_2603_13196_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def _doubles(n, F, T, N):
    """Doubles a build holds: what it needs throughout, the beam, the importance weights, the responses."""
    return 5 * n + 2 * F + 3 * T + n * T + 2 * F * T, n * F * T, 2 * n * F + n, n + N + 1 + N * F * T


def _case(n, F, T):
    return I.make_sky(n, 5), I.make_obs(F, T, 4.0, lst0_h=18.0)


def _same(fg21lib, sky, obs, N, limit, use, **kw):
    ref, kept = fg21lib.fg21_selftest_build_regions(sky, obs, N, 0, **kw)
    got, short = fg21lib.fg21_selftest_build_regions(sky, obs, N, limit, **kw)
    assert (kept, short) == (1, use)
    assert np.array_equal(ref.labels, got.labels) and np.array_equal(ref.edges, got.edges)
    for a, b in zip(fg21lib.fg21_model_get_arrays(ref), fg21lib.fg21_model_get_arrays(got)):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("weighting", ["beam", "sky", "horizon", "uniform"])
def test_no_room_for_the_beam(fg21lib, weighting):
    n, F, T, N = 768, 11, 20, 7
    base, beam, imp, resp = _doubles(n, F, T, N)
    limit = 8 * (base + imp + resp)
    assert 8 * beam > limit // 4
    _same(fg21lib, *_case(n, F, T), N, limit, 0, weighting=weighting)


def test_no_room_for_the_beam_two_weightings(fg21lib):
    n, F, T, N, Na = 768, 11, 20, 5, 3
    base, beam, imp, resp = _doubles(n, F, T, N * Na)
    sky, obs = _case(n, F, T)
    _same(fg21lib, sky, obs, N, 8 * (base + imp + resp), 0, n_alpha=Na, field=I.amplitude_field(sky), weighting_a="sky")


def test_beam_given_back_for_the_importance_weights(fg21lib):
    n, F, T, N = 50, 3, 1, 5
    base, beam, imp, resp = _doubles(n, F, T, N)
    limit = base + imp + n // 2        # room for the weights without the beam, for the responses without the weights
    assert beam <= limit // 4 and base + beam + imp > limit and base + imp + resp > limit
    _same(fg21lib, *_case(n, F, T), N, 8 * limit, 2)


def test_beam_given_back_for_the_responses(fg21lib):
    n, F, T, N = 100, 40, 1, 100
    base, beam, imp, resp = _doubles(n, F, T, N)
    limit = 4 * beam + 200
    assert base + beam + imp <= limit < base + beam + imp + resp
    _same(fg21lib, *_case(n, F, T), N, 8 * limit, 2)


def test_too_little_memory_is_an_error(fg21lib):
    sky, obs = _case(768, 11, 20)
    with pytest.raises(fg21lib.Fg21Error) as e:
        fg21lib.fg21_selftest_build_regions(sky, obs, 7, 200000)
    assert e.value.code == fg21lib.FG21_E_NOMEM
    _, use = fg21lib.fg21_selftest_build_regions(sky, obs, 7)
    assert use == 1
