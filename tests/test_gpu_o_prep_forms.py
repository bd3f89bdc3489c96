"""Prep with the statistics taken by every block (small requests) and by a pass of
their own: the sizes on both sides of the line, points that do not count, and
requests of both kinds in one launch."""
import numpy as np
import pytest

import cases

pytestmark = pytest.mark.gpu


def _model(fg21lib, N, F=7, T=5):
    sky, obs, m, data = cases.small_case(npix=1024, N=N, F=F, T=T, window=3.0)
    model = fg21lib.fg21_build_regions(sky, obs, N)
    fg21lib.fg21_model_set_data(model, data)
    return obs, m, data, model


# up to 256 points and 4096 values (N + 4 a point) take their statistics in every block
@pytest.mark.parametrize("N,P", [(3, 1), (3, 31), (3, 33), (3, 127), (3, 128), (3, 129), (3, 255), (3, 256), (3, 257),
                                 (12, 255), (12, 256), (13, 240), (13, 241), (62, 62), (62, 63)])
def test_statistics_forms(fg21lib, N, P):
    obs, m, data, model = _model(fg21lib, N)
    p = cases.I.prior_draws(P, N, seed=N + P)
    if P > 3:                     # points that do not count: the extremes of the first region lie in them
        p[P // 2, 0], p[P // 2, N + 3] = 9.0, -1.0
        p[P - 1, 0], p[P - 1, N + 1] = -9.0, np.nan
        p[1, N + 2] = 0.0
    got = fg21lib.fg21_loglike_batch(model, p, "fp16x3")
    ok = np.isfinite(p).all(axis=1) & (p[:, N + 3] > 0) & (p[:, N + 2] != 0)
    assert fg21lib.fg21_last_invalid_count() == int((~ok).sum())
    assert np.all(got[~ok] == -np.inf)
    want, _ = cases.expected(m, obs, data, p[ok])
    tol = cases.logl_tolerance("fp16x3", m, obs, data, p[ok])
    assert np.all(np.abs(got[ok] - want) <= tol), cases.fmt_err(f"N{N} P{P}", got[ok], want, tol)


def test_no_valid_point(fg21lib):
    _, _, _, model = _model(fg21lib, 3)
    for P in (5, 300):
        p = cases.I.prior_draws(P, 3, seed=P)
        p[:, 6] = 0.0
        assert np.all(fg21lib.fg21_loglike_batch(model, p, "fp16x3") == -np.inf)


def test_both_forms_in_one_launch(fg21lib):
    models = [_model(fg21lib, N)[3] for N in (3, 12, 5, 20)]
    params = [cases.I.prior_draws(P, m.N, seed=P) for m, P in zip(models, (64, 256, 1000, 300))]
    alone = [fg21lib.fg21_loglike_batch(m, p, "fp16x3") for m, p in zip(models, params)]
    mixed = fg21lib.fg21_loglike_multi(models, params, "fp16x3")
    small = fg21lib.fg21_loglike_multi(models[:2], params[:2], "fp16x3")
    for a, b in zip(alone, mixed):
        assert np.array_equal(a, b)
    for a, b in zip(alone, small):
        assert np.array_equal(a, b)


def test_calls_follow_each_other_over_streams(fg21lib):
    """Calls of one model use one workspace: one made on another stream waits on the GPU."""
    torch = pytest.importorskip("torch")
    _, _, _, model = _model(fg21lib, 9, F=51, T=20)
    ps = [torch.from_numpy(cases.I.prior_draws(P, 9, seed=P)).cuda() for P in (4096, 64, 2000, 129)]
    want = [fg21lib.fg21_loglike_batch(model, p.cpu().numpy(), "fp16x3") for p in ps]
    outs = [torch.empty(len(p), dtype=torch.float64, device="cuda") for p in ps]
    streams = [torch.cuda.Stream() for _ in ps]
    torch.cuda.synchronize()
    for _ in range(20):
        for p, o, s in zip(ps, outs, streams):
            fg21lib.fg21_loglike_batch_device(model, p.data_ptr(), len(p), o.data_ptr(), "fp16x3", s.cuda_stream)
    torch.cuda.synchronize()
    for w, o in zip(want, outs):
        assert np.array_equal(w, o.cpu().numpy())
