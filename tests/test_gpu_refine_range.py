"""The range of the refinement's value and gradient: a PSD value far below the rest outside a candidate's support changes
nothing, inside it the FP64 oracle is met, and whitened data of any finite size give what data of order one give, scaled."""
import numpy as np
import pytest

from oracle import refine
from paper_2110_13115_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

FS, N, F_LOW = 2048.0, 1 << 15, 30.0
MASSES = np.array([(30.0, 25.0), (9.0, 7.0), (29.0, 24.0), (8.0, 7.5)])  # cutoffs of 80, 275, 83 and 284 Hz


@pytest.fixture(scope="module")
def setup():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2110_13115_gb300 import api

    grid = inputs.Grid(FS, N, F_LOW)
    psd = inputs.analytic_psd(grid)
    x = inputs.coloured_noise(grid, psd, 3)
    x = (x + inputs.injection_series(grid, psd, inputs.Injection((9.0, 7.0, 0.0, 0.0), 0.7 * N / FS, 0.4, 20.0), 2)).astype(np.float32)
    s_hat = api.rb_whiten(api.make_desc(FS, N, 1, 1, w=1), torch.from_numpy(x).cuda(), torch.from_numpy(psd).cuda())
    eta = MASSES[:, 0] * MASSES[:, 1] / MASSES.sum(1) ** 2
    theta = np.column_stack([MASSES.sum(1) * eta ** 0.6, np.minimum(eta, 0.2499), 0.7 * N / FS + np.array([0, 1e-3, 0.1, -2.0]),
                             [0.4, -7.0, 3.0, 100.0]])
    return api, psd * 1e-46, s_hat, torch.from_numpy(theta).cuda()  # a PSD in units of strain


def _value_and_gradient(api, s_hat, psd, theta, pn=2):
    d = api.make_refine_desc(FS, N, F_LOW, pn_order=pn, steps=0)
    th = theta.detach().clone().requires_grad_(True)
    J = api.peak_snr2(th, s_hat, torch.from_numpy(psd).cuda(), d)
    J.sum().backward()
    return J.detach(), th.grad


@pytest.mark.parametrize("fill", [1e-130, 1e-300, 5e-324])
@pytest.mark.parametrize("hz", [900.0, 150.0])  # above every cutoff; above the heavy candidates' only
@pytest.mark.parametrize("pn", [2, 3])
def test_small_psd_value_outside_the_support(setup, fill, hz, pn):
    api, psd, s_hat, theta = setup
    J0, g0 = _value_and_gradient(api, s_hat, psd, theta, pn)
    assert (J0 > 0).all() and (g0[:, :3] != 0).all()
    hole = psd.copy()
    hole[int(hz * N / FS)] = fill
    J, g = _value_and_gradient(api, s_hat, hole, theta, pn)
    out = [0, 1, 2, 3] if hz > 300 else [0, 2]
    assert torch.equal(J[out], J0[out]) and torch.equal(g[out], g0[out])
    Jr = api.rb_refine(api.make_refine_desc(FS, N, F_LOW, pn_order=pn, steps=0), s_hat, torch.from_numpy(hole).cuda(), theta)[1]
    assert (Jr - J)[out].abs().max() <= 1e-6 * J[out].max()  # the ascent's FP64 value, to a few FP32 phases


@pytest.mark.parametrize("fill", [1e-60, 1e-130])
def test_small_psd_value_inside_the_support(setup, fill):
    api, psd, s_hat, theta = setup
    hole = psd.copy()
    hole[int(150.0 * N / FS)] = fill
    J, g = _value_and_gradient(api, s_hat, hole, theta)
    s = s_hat.cpu().numpy().astype(np.complex128)
    for i in range(len(theta)):
        th = theta[i].cpu().numpy()
        f, _, amp, sig2 = refine.setup(np.zeros(N // 2 + 1), hole, FS, N, F_LOW, th[0], th[1])
        j = np.rint(f * N / FS).astype(int)
        ws = s[j] * np.sqrt(4.0 * FS / N / hole[j])
        J0, g0 = refine.gradient(th, f, ws, amp, sig2, 2)
        norm = np.sqrt(np.sum(np.abs(ws * amp) ** 2) / sig2)
        # sine and cosine are FP32: 2e-7 a term, so of the norm over the terms
        assert abs(J[i].item() - J0) <= 4e-6 * (np.sqrt(J0) + norm) * max(np.sqrt(J0), 1.0), (i, J0)
        if J0 > 25.0:
            assert np.all(np.abs(g[i].cpu().numpy() - g0) <= 1e-3 * np.abs(g0) + 1e-5 * np.linalg.norm(g0)), (i, g[i], g0)


@pytest.mark.parametrize("power", [-80, 110])
def test_size_of_the_data(setup, power):
    api, psd, s_hat, theta = setup
    J0, g0 = _value_and_gradient(api, s_hat, psd, theta)
    J, g = _value_and_gradient(api, s_hat * 2.0 ** power, psd, theta)
    assert torch.equal(J, J0 * 4.0 ** power) and torch.equal(g, g0 * 4.0 ** power)


def test_infinite_value(setup):
    api, psd, s_hat, theta = setup
    J0, _ = _value_and_gradient(api, s_hat, psd, theta)
    bad = s_hat.clone()
    bad[int(150.0 * N / FS)] = complex(float("inf"), 0.0)  # in the light candidates' supports
    J, _ = _value_and_gradient(api, bad, psd, theta)
    assert torch.equal(J[[0, 2]], J0[[0, 2]]) and torch.isinf(J[[1, 3]]).all()
