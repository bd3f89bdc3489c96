"""A stream under capture is refused before anything is allocated, waited for or
enqueued, and the caller's capture stays intact."""
import numpy as np
import pytest

import cases

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("warm", [False, True])       # the model's workspace not made yet, and made but too small
@pytest.mark.parametrize("call", ["device", "host", "multi", "eval", "autotune"])
def test_capturing_stream_is_refused(fg21lib, call, warm):
    torch = pytest.importorskip("torch")
    sky, obs, m, data = cases.small_case(npix=1024, N=3, F=7, T=5, window=3.0)
    model = fg21lib.fg21_build_regions(sky, obs, 3)
    fg21lib.fg21_model_set_data(model, data)
    p = cases.I.prior_draws(3000, 3, seed=1)
    d_p = torch.from_numpy(p).cuda()
    d_l = torch.full((len(p),), 7.0, dtype=torch.float64, device="cuda")
    if warm:
        fg21lib.fg21_loglike_batch(model, p[:64], "fp16x3")
    s = torch.cuda.Stream()
    h = s.cuda_stream
    go = {"device": lambda: fg21lib.fg21_loglike_batch_device(model, d_p.data_ptr(), len(p), d_l.data_ptr(), "fp16x3", h),
          "host": lambda: fg21lib.fg21_loglike_batch(model, p, "fp16x3", h),
          "multi": lambda: fg21lib.fg21_loglike_multi([model], [p], "fp16x3", h),
          "eval": lambda: fg21lib.fg21_model_eval(model, p[:4], "fp16x3", h),
          "autotune": lambda: fg21lib.fg21_autotune(model, d_p.data_ptr(), len(p), d_l.data_ptr(), "fp16x3", h)}[call]
    x = torch.zeros(8, device="cuda")
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s, capture_error_mode="thread_local"):
        x.add_(1)
        with pytest.raises(fg21lib.Fg21Error, match="captured") as e:
            go()
        x.add_(1)
    assert e.value.code == fg21lib.FG21_E_CUDA
    g.replay()
    torch.cuda.synchronize()
    assert torch.all(x == 2) and torch.all(d_l == 7.0)     # the capture holds the caller's own work and nothing else
    got = fg21lib.fg21_loglike_batch(model, p, "fp16x3")
    want, _ = cases.expected(m, obs, data, p)
    assert np.all(np.abs(got - want) <= cases.logl_tolerance("fp16x3", m, obs, data, p))
