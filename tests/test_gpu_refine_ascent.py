"""The ascent, whose candidates are shared among the CTAs of a cluster: a candidate's result is the same bits in any
company, refused candidates leave alone, and no step gives the value that the evaluation gives."""
import numpy as np
import pytest

from paper_2110_13115_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

@pytest.mark.parametrize("n,f_low,pn,count", [
    (1 << 10, 30.0, 2, 1),  # fewer frequencies than threads for the heavy ones
    (1 << 14, 16.0, 0, 3),
    (1 << 15, 31.9375, 3, 40),
    (1 << 18, 20.0, 2, 700),  # more candidates than fit the chip at once
])
def test_ascent(n, f_low, pn, count):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2110_13115_gb300 import api

    fs = 2048.0
    grid = inputs.Grid(fs, n, f_low)
    psd = inputs.analytic_psd(grid)
    x = inputs.coloured_noise(grid, psd, 5)
    inj = inputs.Injection((9.0, 7.0, 0.0, 0.0), 0.7 * n / fs, 0.4, 20.0)
    x = (x + inputs.injection_series(grid, psd, inj, max(pn, 2))).astype(np.float32)
    psd_d = torch.from_numpy(psd).cuda()
    s_hat = api.rb_whiten(api.make_desc(fs, n, 1, 1, w=1), torch.from_numpy(x).cuda(), psd_d)
    rng = np.random.default_rng(count)
    theta = np.column_stack([rng.uniform(6.0, 40.0, count), rng.uniform(0.15, 0.25, count),
                             0.7 * n / fs + rng.normal(0, 1e-2, count), rng.uniform(-3, 3, count)])
    theta[0, 1] = 0.25
    th = torch.from_numpy(theta).cuda()
    d = api.make_refine_desc(fs, n, f_low, pn_order=pn, steps=4)
    t, J = api.rb_refine(d, s_hat, psd_d, th)
    assert torch.isfinite(J).all() and torch.isfinite(t).all()
    for i in {0, count // 2, count - 1}:
        ti, Ji = api.rb_refine(d, s_hat, psd_d, th[i : i + 1])
        assert torch.equal(ti[0], t[i]) and torch.equal(Ji[0], J[i])
    # no step: the evaluation's value; its terms are the same to a few FP32 phases of a last digit (1e-7 of a term)
    t0, J0 = api.rb_refine(api.make_refine_desc(fs, n, f_low, pn_order=pn, steps=0), s_hat, psd_d, th)
    Je, _ = api.rb_refine_eval(d, s_hat, psd_d, th)
    assert torch.allclose(t0, th, rtol=4e-16, atol=0.0)  # (scaled and back)
    assert (J0 - Je).abs().max() <= 1e-6 * Je.max()
    assert (J >= J0).all()
    bad = th.clone()
    bad[count // 2, 1] = 0.3
    with pytest.raises(Exception, match="eta outside"):
        api.rb_refine(d, s_hat, psd_d, bad)
