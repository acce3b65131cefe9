"""The gradient's sums are at least as precise as sums in FP64: Z as the adjoint forms it (values in three FP32 parts)
against the ascent's FP64 value of the same phases, sines and cosines."""
import numpy as np
import pytest

from oracle import refine
from paper_2110_13115_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,pn", [(1 << 13, 0), (1 << 14, 2), (1 << 15, 3)])
def test_sums_against_fp64(n, pn):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2110_13115_gb300 import api

    fs, f_low, T = 2048.0, 30.0, 64
    grid = inputs.Grid(fs, n, f_low)
    psd = inputs.analytic_psd(grid) * 1e-46
    rng = np.random.default_rng(n)
    s = (rng.standard_normal(n // 2) + 1j * rng.standard_normal(n // 2)).astype(np.complex64)
    theta = np.column_stack([rng.uniform(7.0, 12.0, T), rng.uniform(0.2, 0.2499, T), 0.7 * n / fs + rng.normal(0, 1e-2, T),
                             rng.uniform(-3, 3, T)])
    s_d, psd_d, th = torch.from_numpy(s).cuda(), torch.from_numpy(psd).cuda(), torch.from_numpy(theta).cuda()
    d = api.make_refine_desc(fs, n, f_low, pn_order=pn, steps=0)
    J64 = api.rb_refine(d, s_d, psd_d, th)[1].cpu().numpy()
    one = torch.ones(T, dtype=torch.float64, device="cuda")
    # dJ/dphi_c at a given Z is 2 Im(conj(Z) Z') / sigma^2: Z = 1 and i give both parts of the adjoint's own sum Z'
    part = [api.rb_refine_adjoint(d, s_d, psd_d, th, torch.full((T,), z, dtype=torch.complex128, device="cuda"), one)[:, 3]
            .cpu().numpy().astype(np.longdouble) for z in (1.0, 1j)]
    err = []
    for i in range(T):
        f, _, amp, _ = refine.setup(np.zeros(n // 2 + 1), psd, fs, n, f_low, theta[i, 0], theta[i, 1])
        j = np.rint(f * n / fs).astype(int)
        a2 = f.astype(np.longdouble) ** (np.longdouble(-7) / 3) * (np.longdouble(4 * fs / n) / psd[j])
        sig2 = a2.sum()
        norm2 = (a2 * np.abs(s[j].astype(np.complex128)) ** 2).sum() / sig2
        J = (part[0][i] ** 2 + part[1][i] ** 2) * sig2 / 4
        err.append(float((J - J64[i]) / (2 * np.sqrt(J * norm2))))  # of Z along itself, relative to the norm of its terms
    # FP64: a chain of some ten additions a thread and eight warps, two or three roundings a term: under 4 units of 2^-53
    # of the norm; the three parts: the rounding of amp and of the final value, under 2
    assert np.sqrt(np.mean(np.square(err))) <= 6 * 2.0 ** -53
