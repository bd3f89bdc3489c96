"""Calls of one model share one workspace: a call on another stream waits on the
GPU for the one before it.  Every call of every round has an output of its own,
filled beforehand, and all are compared."""
import numpy as np
import pytest

import cases

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["fp16x3", "fp32_delta"])
def test_every_call_over_streams(fg21lib, prec):
    torch = pytest.importorskip("torch")
    sky, obs, m, data = cases.small_case(npix=1024, N=9, F=51, T=20, window=3.0)
    model = fg21lib.fg21_build_regions(sky, obs, 9)
    fg21lib.fg21_model_set_data(model, data)
    ps = [torch.from_numpy(cases.I.prior_draws(P, 9, seed=P)).cuda() for P in (4096, 64, 2000, 129)]
    want = [fg21lib.fg21_loglike_batch(model, p.cpu().numpy(), prec) for p in ps]
    rounds = 20
    outs = [[torch.full((len(p),), float("nan"), dtype=torch.float64, device="cuda") for p in ps] for _ in range(rounds)]
    streams = [torch.cuda.Stream() for _ in ps]
    torch.cuda.synchronize()
    for r in range(rounds):
        for k in np.random.default_rng(r).permutation(len(ps)):
            fg21lib.fg21_loglike_batch_device(model, ps[k].data_ptr(), len(ps[k]), outs[r][k].data_ptr(), prec,
                                              streams[k].cuda_stream)
    torch.cuda.synchronize()
    for r in range(rounds):
        for k, w in enumerate(want):
            assert np.array_equal(w, outs[r][k].cpu().numpy()), (r, k)
