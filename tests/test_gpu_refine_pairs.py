"""The refinement's FP32-pair arithmetic against FP64: long phases, every phase order, edges of the chunks over
which sigma^2 is summed, and PSDs in strain units far outside the range of FP32."""
import numpy as np
import pytest

from oracle import mf, refine
from paper_2110_13115_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def api():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2110_13115_gb300 import api as A

    return A


@pytest.mark.parametrize("n,f_low,pn,scale", [
    (1 << 10, 30.0, 2, 1.0),  # a handful of frequencies
    (1 << 14, 16.0, 0, 1e-46),  # band from a chunk's first frequency, strain units
    (1 << 15, 31.9375, 3, 1.0),  # band within a chunk
    (1 << 18, 20.0, 3, 1e120),
])
def test_pairs_against_fp64(api, n, f_low, pn, scale):
    fs = 2048.0
    grid = inputs.Grid(fs, n, f_low)
    psd = inputs.analytic_psd(grid)
    x = inputs.coloured_noise(grid, psd, 3)
    inj = inputs.Injection((9.0, 7.0, 0.0, 0.0), 0.7 * n / fs, 0.4, 20.0)
    x = (x + inputs.injection_series(grid, psd, inj, max(pn, 2))).astype(np.float32)
    s_fd = mf.strain_fd(x.astype(np.float64), fs)
    psd_d = torch.from_numpy(psd).cuda()
    s_hat = api.rb_whiten(api.make_desc(fs, n, 1, 1, w=1), torch.from_numpy(x).cuda(), psd_d)
    m = np.array([(9.0, 7.0), (1.4, 1.3), (40.0, 25.0), (9.01, 6.99)])
    eta = m[:, 0] * m[:, 1] / m.sum(1) ** 2
    theta = np.column_stack([m.sum(1) * eta ** 0.6, np.minimum(eta, 0.2499), 0.7 * n / fs + np.array([0, 1e-3, 0.1, -2.0]),
                             [0.4, -7.0, 3.0, 100.0]])
    d = api.make_refine_desc(fs, n, f_low, pn_order=pn, steps=0)
    # J and its gradient are what they are in units where the PSD is of order one
    th = torch.from_numpy(theta).cuda().requires_grad_(True)
    J = api.peak_snr2(th, s_hat, psd_d * scale, d)
    J.sum().backward()
    got = th.grad.cpu().numpy()
    _, Z = api.rb_refine_eval(d, s_hat, psd_d * scale, th.detach())
    assert np.all(np.isfinite(Z.cpu().numpy()))
    # s_hat is FP32 (about 5e-7 of its norm); sine and cosine are FP32: 2e-7 a term, so of the norm over the terms
    for i in range(len(theta)):
        f, ws, amp, sig2 = refine.setup(s_fd, psd, fs, n, f_low, theta[i, 0], theta[i, 1])
        if len(f) == 0:
            continue
        J0, g0 = refine.gradient(theta[i], f, ws, amp, sig2, pn)
        norm = np.sqrt(np.sum(np.abs(ws * amp) ** 2) / sig2)  # |Z| of incoherent terms, in SNR units
        tol = 4e-6 * (np.sqrt(J0) + norm) * max(np.sqrt(J0), 1.0)
        assert abs(J.detach().cpu().numpy()[i] - J0) <= tol, (i, J0)
        if J0 > 25.0:
            assert np.all(np.abs(got[i] - g0) <= 1e-3 * np.abs(g0) + 1e-5 * np.linalg.norm(g0)), (i, got[i], g0)
