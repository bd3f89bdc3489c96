"""The allocation-free call gives the regular call's results bit for bit, also
where the partial sums of all points do not fit its scratch and the points go in
parts (the sizes lie between the regular split's need and the call's limit)."""
import numpy as np
import pytest

import cases

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,F,T,P", [(24, 301, 100, 70000),     # one part
                                     (24, 301, 100, 72300), (24, 301, 100, 95230), (41, 211, 217, 41470),
                                     (5, 51, 10, 173312)])
@pytest.mark.parametrize("prec", ["fp16x3", "bf16x3"])
def test_same_bits_at_the_limit(fg21lib, N, F, T, P, prec):
    torch = pytest.importorskip("torch")
    sky, obs, m, data = cases.small_case(npix=1024, N=N, F=F, T=T, window=3.0)
    model = fg21lib.fg21_build_regions(sky, obs, N)
    fg21lib.fg21_model_set_data(model, data)
    p = cases.I.prior_draws(P, N, seed=P)
    p[P // 2, N + 3] = 0.0                    # points that do not count, in the middle and at the end
    p[P - 1, N + 2] = 0.0
    d_p = torch.from_numpy(p).cuda()
    d_l = torch.full((P,), float("nan"), dtype=torch.float64, device="cuda")
    d_n = torch.full((P + 128,), 7.0, dtype=torch.float64, device="cuda")
    s = torch.cuda.current_stream().cuda_stream
    fg21lib.fg21_loglike_batch_device(model, d_p.data_ptr(), P, d_l.data_ptr(), prec, s)
    for _ in range(2):
        fg21lib.fg21_loglike_batch_device_noalloc(model, d_p.data_ptr(), P, d_n.data_ptr(), prec, s)
        torch.cuda.synchronize()
        want, got = d_l.cpu().numpy(), d_n.cpu().numpy()
        assert np.isneginf(want).sum() == 2 and not np.isnan(want).any()
        assert np.array_equal(want, got[:P]) and np.all(got[P:] == 7.0)
        d_n.fill_(7.0)


def test_parts_under_capture(fg21lib):
    """The call may be captured (after a first call on the device); a replay runs the parts again."""
    torch = pytest.importorskip("torch")
    sky, obs, m, data = cases.small_case(npix=1024, N=5, F=51, T=10, window=3.0)
    model = fg21lib.fg21_build_regions(sky, obs, 5)
    fg21lib.fg21_model_set_data(model, data)
    P = 173312
    d_p = torch.from_numpy(cases.I.prior_draws(P, 5, seed=1)).cuda()
    d_l = torch.full((P,), float("nan"), dtype=torch.float64, device="cuda")
    d_n = torch.full((P,), float("nan"), dtype=torch.float64, device="cuda")
    s = torch.cuda.Stream()
    fg21lib.fg21_loglike_batch_device(model, d_p.data_ptr(), P, d_l.data_ptr(), "fp16x3", 0)
    fg21lib.fg21_loglike_batch_device_noalloc(model, d_p.data_ptr(), P, d_n.data_ptr(), "fp16x3", 0)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s, capture_error_mode="thread_local"):
        fg21lib.fg21_loglike_batch_device_noalloc(model, d_p.data_ptr(), P, d_n.data_ptr(), "fp16x3", s.cuda_stream)
    for _ in range(2):
        d_n.fill_(float("nan"))
        g.replay()
        torch.cuda.synchronize()
        assert torch.equal(d_n, d_l)
