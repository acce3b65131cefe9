"""The fused four-step transforms at the edges of their range: every column length from 128 points, more rows than
the ring holds, rows and outputs on 8-byte boundaries only, no beta, and the folded spectra of each width."""
import numpy as np
import pytest

from oracle import mf, rb
from paper_2110_13115_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def api():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2110_13115_gb300 import api as A

    return A


def _block(n, seed=5):
    grid = inputs.Grid(2048.0, n, 30.0)
    psd = inputs.analytic_psd(grid)
    return psd, inputs.coloured_noise(grid, psd, seed).astype(np.float32)


def _rows(k, half, seed, offset=0):
    """Unit rows on the device, their first value `offset` complex numbers into an allocation."""
    p = inputs.unit_rows(k, half, seed).astype(np.complex64)
    buf = torch.empty(k * half + offset, dtype=torch.complex64, device="cuda")
    buf[offset:] = torch.from_numpy(p.reshape(-1)).cuda()
    return p, buf[offset:].view(k, half)


# the fused launch takes over at 2^23 points (2^22 from 2^17 samples); ring lengths are at most 512 rows of 2^14, 128 of
# 2^16 and 16 of 2^19 samples
@pytest.mark.parametrize("n,k,w,offset", [(1 << 14, 512, 16, 0), (1 << 14, 511, 16, 0), (1 << 14, 700, 1, 1), (1 << 15, 257, 2, 0), (1 << 16, 300, 4, 0),
                                          (1 << 17, 33, 8, 1), (1 << 18, 16, 16, 1), (1 << 19, 40, 8, 0), (1 << 20, 4, 16, 0)])
def test_basis_series(api, n, k, w, offset):
    half, fs = n // 2, 2048.0
    psd, x = _block(n)
    p, rows = _rows(k, half, 7, offset)
    d = api.make_desc(fs, n, k, 1, w=w)
    basis = api.Basis(rows, torch.ones((1, k), dtype=torch.complex64, device="cuda"), n)
    sh = api.rb_whiten(d, torch.from_numpy(x).cuda(), torch.from_numpy(psd).cuda())
    beta, bavg = api.rb_basis_filter(d, basis, sh)
    again, avg2 = api.rb_basis_filter(d, basis, sh, keep_beta=False)
    assert again is None and torch.equal(avg2, bavg)
    s64 = sh.to(torch.complex128)
    for r0 in range(0, k, 64):
        ref = (torch.fft.ifft(s64 * rows[r0:r0 + 64].to(torch.complex128).conj(), n=n) * n)[:, half:]
        scale = ref.abs().square().mean().sqrt()
        # FP32 transform of log2 n <= 20 levels and three twiddle products: within 20 * 4 * 2^-24 of the rms
        assert (beta[r0:r0 + 64] - ref).abs().max() / scale < 1e-5
        assert (bavg[r0:r0 + 64] - ref.view(len(ref), -1, w).mean(2)).abs().max() / scale < 1e-5


@pytest.mark.parametrize("n,w,T,rho", [(1 << 14, 1, 513, 3.9), (1 << 14, 16, 512, 0.0), (1 << 15, 8, 256, 3.0), (1 << 17, 2, 32, 3.5),
                                       (1 << 20, 16, 4, 3.5), (1 << 20, 16, 3, 3.5)])
def test_template_windows(api, n, w, T, rho):
    fs = 2048.0
    psd, x = _block(n, 6)
    p, rows = _rows(T, n // 2, 8, 1)
    d = api.make_desc(fs, n, 1, T, w=w, rho_ii=rho)
    buf, nt = api.rb_filter_plain(d, rows, torch.from_numpy(x).cuda(), torch.from_numpy(psd).cuda())
    got = api.triggers_numpy(buf, nt)
    z = rb.basis_series(mf.strain_fd(x.astype(np.float64), fs), psd, p.astype(np.complex128), n, fs)[:, n // 2:]
    best = np.abs(z).reshape(T, -1, w).max(axis=2)
    if rho == 0.0:
        assert nt == best.size
    key = got["tmpl"].astype(np.int64) * (n // w) + got["sample"] // w - n // (2 * w)
    assert len(np.unique(key)) == nt
    t, b = got["tmpl"], got["sample"] // w - n // (2 * w)
    assert np.all(np.abs(got["snr"] - best[t, b]) <= 1e-5 * np.abs(z).max())
    assert np.all(np.abs(np.abs(z[t, got["sample"] - n // 2]) - best[t, b]) <= 2e-5 * np.abs(z).max())
    seen = np.zeros(best.shape, bool)
    seen[t, b] = True
    assert np.all(seen[best > rho * 1.0001]) and not np.any(seen[best < rho * 0.9999])


@pytest.mark.parametrize("n,w,T,offset", [(1 << 15, 2, 512, 0), (1 << 15, 2, 511, 0), (1 << 16, 4, 513, 1), (1 << 18, 16, 600, 0),
                                          (1 << 19, 2, 20, 1), (1 << 19, 8, 130, 1)])
def test_folded_spectra(api, n, w, T, offset):
    fs, rho = 2048.0, 3.5
    psd, x = _block(n, 9)
    p, rows = _rows(T, n // 2, 10, offset)
    psd_d, x_d = torch.from_numpy(psd).cuda(), torch.from_numpy(x).cuda()
    d = api.make_desc(fs, n, 1, T, w=w, rho_i=rho, cand_capacity=1 << 22)
    s64 = api.rb_whiten(d, x_d, psd_d).to(torch.complex128)
    for entry, lowpass in ((api.rb_stage1_folded, False), (api.rb_stage1_lowpass, True)):
        c = api.candidates_numpy(*entry(d, rows, x_d, psd_d))
        seen = np.zeros((T, n // (2 * w)), bool)
        snr = np.zeros(seen.shape)
        seen[c["tmpl"], c["bin"] - n // (2 * w)] = True
        snr[c["tmpl"], c["bin"] - n // (2 * w)] = c["snr_avg"]
        for t in range(T):
            q = s64 * rows[t].to(torch.complex128).conj()
            if lowpass:
                z = (torch.fft.ifft(q[: n // w]) * (n // w))[n // (2 * w):].abs().cpu().numpy()
            else:
                z = (torch.fft.ifft(q, n=n) * n)[n // 2:].view(-1, w).mean(1).abs().cpu().numpy()
            assert np.all(seen[t][z > rho * 1.0001]) and not np.any(seen[t][z < rho * 0.9999])
            assert np.all(np.abs(snr[t] - z)[seen[t]] <= 1e-5 * max(z.max(), 1.0))
