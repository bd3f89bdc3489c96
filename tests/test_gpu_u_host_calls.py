"""The host-buffer call by direct launches (first call of a size) and by the kept
graph (later ones), to pageable and page-locked buffers, on both sides of the
size up to which a page-locked result comes by way of the staging buffer: the
same logL, and the invalid count of each call."""
import numpy as np
import pytest

import cases

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["fp16x3", "fp32_delta"])
@pytest.mark.parametrize("P", [1, 31, 500, 2047, 2048, 2049, 5000])
def test_host_call_forms(fg21lib, P, prec):
    torch = pytest.importorskip("torch")
    sky, obs, m, data = cases.small_case(npix=1024, N=5, F=21, T=7, window=3.0)
    model = fg21lib.fg21_build_regions(sky, obs, 5)
    fg21lib.fg21_model_set_data(model, data)
    other = cases.I.prior_draws(77, 5, seed=77)
    want_other = fg21lib.fg21_loglike_batch(model, other, prec)
    d_l = torch.empty(P, dtype=torch.float64, device="cuda")
    for k in range(6):
        p = cases.I.prior_draws(P, 5, seed=100 * P + k)
        p[: k % 3, 8] = 0.0                                  # 0, 1 or 2 points that do not count
        bad = min(P, k % 3)
        d_p = torch.from_numpy(p).cuda()
        fg21lib.fg21_loglike_batch_device(model, d_p.data_ptr(), P, d_l.data_ptr(), prec, 0)
        want = d_l.cpu().numpy()
        for locked in (False, True):
            out = torch.full((P,), 7.0, dtype=torch.float64)
            src = torch.from_numpy(p)
            if locked:
                out, src = out.pin_memory(), src.pin_memory()
            got = fg21lib.fg21_loglike_batch(model, src.numpy(), prec, out=out.numpy())
            assert fg21lib.fg21_last_invalid_count() == bad
            assert np.array_equal(got, want) and np.isneginf(got).sum() == bad
        if k == 3:                                           # a call of another size in between
            assert np.array_equal(fg21lib.fg21_loglike_batch(model, other, prec), want_other)
