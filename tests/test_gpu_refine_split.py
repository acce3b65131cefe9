"""Value and adjoint with a candidate's frequencies shared among the CTAs of a cluster (few candidates) against one CTA
per candidate (many): the same terms, summed in another order."""
import numpy as np
import pytest

from paper_2110_13115_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,pn,few", [
    (1 << 10, 2, 1),  # too short to share
    (1 << 14, 3, 3),  # two CTAs leave a thread 32 frequencies of the block
    (1 << 16, 0, 64),  # the last count for eight CTAs, the first and last for four, for two
    (1 << 16, 2, 65),
    (1 << 16, 3, 128),
    (1 << 16, 2, 129),
    (1 << 17, 2, 256),
])
def test_split_against_whole(n, pn, few):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2110_13115_gb300 import api

    fs, f_low, many = 2048.0, 30.0, 1000
    grid = inputs.Grid(fs, n, f_low)
    psd = inputs.analytic_psd(grid)
    x = inputs.coloured_noise(grid, psd, 5)
    inj = inputs.Injection((9.0, 7.0, 0.0, 0.0), 0.7 * n / fs, 0.4, 20.0)
    x = (x + inputs.injection_series(grid, psd, inj, max(pn, 2))).astype(np.float32)
    psd_d = torch.from_numpy(psd).cuda()
    s_hat = api.rb_whiten(api.make_desc(fs, n, 1, 1, w=1), torch.from_numpy(x).cuda(), psd_d)
    rng = np.random.default_rng(few)
    theta = np.column_stack([rng.uniform(6.5, 7.5, many), rng.uniform(0.15, 0.2499, many),
                             0.7 * n / fs + rng.normal(0, 1e-2, many), rng.uniform(-3, 3, many)])
    th = torch.from_numpy(theta).cuda()
    d = api.make_refine_desc(fs, n, f_low, pn_order=pn, steps=0)
    J1, Z1 = api.rb_refine_eval(d, s_hat, psd_d, th[:few])
    J2, Z2 = api.rb_refine_eval(d, s_hat, psd_d, th)
    # sums of equal terms in another order: a few 1e-15 of their norm, taken as 1e-11 of the largest result
    assert (Z1 - Z2[:few]).abs().max() <= 1e-11 * Z2.abs().max()
    assert (J1 - J2[:few]).abs().max() <= 1e-11 * J2.max()
    dJ = torch.ones(many, dtype=torch.float64, device="cuda")
    g1 = api.rb_refine_adjoint(d, s_hat, psd_d, th[:few], Z1, dJ[:few])
    g2 = api.rb_refine_adjoint(d, s_hat, psd_d, th, Z2, dJ)
    for k in range(3):
        assert (g1 - g2[:few])[:, k].abs().max() <= 1e-9 * g2[:, k].abs().max()
    assert (g1 - g2[:few])[:, 3].abs().max() <= 1e-9 * J2.max()  # (zero but for rounding)
    if few > 1:  # a refused candidate's CTAs leave, the others go on
        bad = th[:few].clone()
        bad[few // 2, 1] = 0.3
        with pytest.raises(Exception, match="eta outside"):
            api.rb_refine_eval(d, s_hat, psd_d, bad)
