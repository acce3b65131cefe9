"""Value and gradient of a candidate are the same bits in any company: one CTA per candidate and two, four or eight of them
sum the same strands in the same order."""
import numpy as np
import pytest

from paper_2110_13115_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,f_low,pn", [
    (1 << 10, 30.0, 2),  # one strand
    (1 << 14, 16.0, 3),  # two
    (1 << 15, 31.9375, 0),  # four
    (1 << 16, 30.0, 3),  # eight, some of them empty for the heaviest
    (1 << 18, 20.0, 2),
])
def test_company(n, f_low, pn):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2110_13115_gb300 import api

    fs, many = 2048.0, 700
    grid = inputs.Grid(fs, n, f_low)
    psd = inputs.analytic_psd(grid)
    x = inputs.coloured_noise(grid, psd, 5).astype(np.float32)
    psd_d = torch.from_numpy(psd).cuda()
    s_hat = api.rb_whiten(api.make_desc(fs, n, 1, 1, w=1), torch.from_numpy(x).cuda(), psd_d)
    rng = np.random.default_rng(n)
    theta = np.column_stack([rng.uniform(6.0, 60.0, many), rng.uniform(0.15, 0.25, many),
                             0.7 * n / fs + rng.normal(0, 1e-2, many), rng.uniform(-3, 3, many)])
    th = torch.from_numpy(theta).cuda()
    d = api.make_refine_desc(fs, n, f_low, pn_order=pn, steps=0)
    J, Z = api.rb_refine_eval(d, s_hat, psd_d, th)
    dJ = torch.linspace(0.5, 2.0, many, dtype=torch.float64, device="cuda")
    g = api.rb_refine_adjoint(d, s_hat, psd_d, th, Z, dJ)
    for count in (1, 64, 65, 128, 129, 256, 257):  # the last counts for eight, four and two CTAs, and the next ones
        c = slice(many - count, many)
        Jc, Zc = api.rb_refine_eval(d, s_hat, psd_d, th[c])
        gc = api.rb_refine_adjoint(d, s_hat, psd_d, th[c], Z[c], dJ[c])
        # (by their bits: an empty support gives NaN)
        for one, all_ in ((Jc, J[c]), (torch.view_as_real(Zc), torch.view_as_real(Z[c])), (gc, g[c])):
            assert torch.equal(one.contiguous().view(torch.int64), all_.contiguous().view(torch.int64)), count
