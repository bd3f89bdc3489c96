"""The tensor kernel's forms against the oracle, at the edges of each choice it
makes: the code for every count of region chunks (K and the trough's place
change there) with every series degree, every count of column blocks, and the
work items spread over the two lanes of a CTA."""
import numpy as np
import pytest

import cases

pytestmark = pytest.mark.gpu


def _check(fg21lib, N, F, T, params, npix=1024):
    sky, obs, m, data = cases.small_case(npix=npix, N=N, F=F, T=T, window=3.0)
    model = fg21lib.fg21_build_regions(sky, obs, N)
    fg21lib.fg21_model_set_data(model, data)
    for p in params:
        got = fg21lib.fg21_loglike_batch(model, p, "fp16x3")
        want, _ = cases.expected(m, obs, data, p)
        tol = cases.logl_tolerance("fp16x3", m, obs, data, p)
        assert np.all(np.abs(got - want) <= tol), cases.fmt_err(f"N{N} F{F} T{T} P{len(p)}", got, want, tol)


@pytest.mark.parametrize("N", [1, 8, 9, 14, 15, 16, 17, 24, 25, 30, 31, 32, 33, 40, 41, 46, 47, 48, 49, 56, 57, 62])
def test_region_chunks(fg21lib, N):
    # largest |expm1 argument| about 1.5 times the spread: degrees 3, 5, 8, then 8 with squarings
    theta = cases.I.prior_draws(1, N, seed=N)[0]
    theta[:N], theta[N + 3] = 2.6, cases.I.NOISE_K
    _check(fg21lib, N, 5, 3, [cases.I.scatter_around(theta, 130, s, seed=N, d21=0.1) for s in (1e-4, 0.03, 0.3, 1.0)])


@pytest.mark.parametrize("T", [1, 16, 17, 33, 49, 65, 81, 97, 113, 129, 145, 161, 177, 192, 193, 385])
def test_column_blocks(fg21lib, T):
    _check(fg21lib, 5, 3, T, [cases.I.prior_draws(P, 5, seed=T) for P in (1, 128, 129)])


@pytest.mark.parametrize("tiles", [1, 151, 152, 153, 304, 305, 457])
def test_items_over_lanes(fg21lib, tiles):
    # one channel: a work item per 128-point tile, so the lanes of 152 CTAs hold none, one or several
    _check(fg21lib, 3, 1, 2, [cases.I.prior_draws(128 * tiles - 5, 3, seed=tiles)])


def test_items_of_other_widths_follow_each_other(fg21lib):
    """Items with other numbers of columns, one after the other in a lane, use one
    accumulator: what one still reads, the next must not write."""
    models, params = [], []
    for k, T in enumerate((10, 97, 33, 129, 1, 64, 177, 17, 80, 48)):
        N = 3 + 4 * (k % 4)
        sky, obs, m, data = cases.small_case(npix=1024, N=N, F=31, T=T, window=3.0)
        model = fg21lib.fg21_build_regions(sky, obs, N)
        fg21lib.fg21_model_set_data(model, data)
        models.append(model)
        params.append(cases.I.prior_draws(2500 - 130 * k, N, seed=k))
    alone = [fg21lib.fg21_loglike_batch(m, p, "fp16x3") for m, p in zip(models, params)]
    for rep in range(30):
        order = np.random.default_rng(rep).permutation(len(models))
        mixed = fg21lib.fg21_loglike_multi([models[i] for i in order], [params[i] for i in order], "fp16x3")
        for i, got in zip(order, mixed):
            assert np.array_equal(alone[i], got), (rep, models[i].T, int(np.sum(alone[i] != got)))
