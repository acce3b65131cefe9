"""The fused transforms against the two radix-16 passes at the counts of rows where the one takes over from the other, at
every length, bin width and kind of rows. Which of the two ran is seen from the launches (basis filter) or from last bits."""
import pytest

from paper_2110_13115_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

LENGTHS = [1 << p for p in range(14, 21)]
# both are FP32 transforms of at most 20 levels and three twiddle products: 20 * 4 * 2^-24 of the rms each
TOL = 1e-5


def _line(n, w):
    """The first count of rows that takes the fused launch."""
    return (1 << 22 if n >= 1 << 17 else 3 << 22 if n == 1 << 14 and w == 1 else 1 << 23) // n


def _fold_line(m, lowpass):
    """The same for the folded first stage and the one without a fold, which takes it at 2^19 points only."""
    return (1 << 23 if lowpass else 1 << 22 if m == 1 << 14 else 1 << 21) // m


@pytest.fixture(scope="module")
def env():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2110_13115_gb300 import _native as N, api

    lib = N.load()
    yield api, lib
    lib.rbx_set_fft_radix32(1)


def _both(env, call):
    """call() by the fused launch and by the passes, with the launches that each took."""
    api, lib = env
    out = []
    for mode in (1, 0):
        lib.rbx_set_fft_radix32(mode)
        before = api.rb_kernel_launches()
        res = call()
        out.append((res, api.rb_kernel_launches() - before))
    lib.rbx_set_fft_radix32(1)
    return out


def _rows(k, half, seed):
    g = torch.Generator("cuda").manual_seed(seed)
    x = torch.view_as_complex(torch.randn((k, half, 2), generator=g, device="cuda"))
    return x / half ** 0.5


def _strain(n):
    grid = inputs.Grid(2048.0, n, 30.0)
    psd = inputs.analytic_psd(grid)
    x = inputs.coloured_noise(grid, psd, 5).astype("float32")
    return torch.from_numpy(x).cuda(), torch.from_numpy(psd).cuda()


@pytest.mark.parametrize("n", LENGTHS)
@pytest.mark.parametrize("w", [1, 2, 4, 8, 16])
def test_basis_filter(env, n, w):
    api = env[0]
    sh = _rows(1, n // 2, 1)[0] * (n // 2) ** 0.5
    for k, fused in ((_line(n, w), True), (_line(n, w) + 1, True), (_line(n, w) - 1, False)):
        rows = _rows(k, n // 2, 2)
        d = api.make_desc(2048.0, n, k, 1, w=w)
        basis = api.Basis(rows, torch.ones((1, k), dtype=torch.complex64, device="cuda"), n)
        ((beta, avg), one), ((beta0, avg0), two) = _both(env, lambda: api.rb_basis_filter(d, basis, sh))
        assert (one == 2) == fused and two >= 3  # (the tables are one of them)
        if not fused:
            assert torch.equal(beta, beta0) and torch.equal(avg, avg0)
        for a, b in ((beta, beta0), (avg, avg0)):
            assert (a - b).abs().max() <= 2 * TOL * beta0.abs().square().mean().sqrt()


@pytest.mark.parametrize("n", LENGTHS)
@pytest.mark.parametrize("w", [1, 8, 16])
def test_template_method(env, n, w):
    api = env[0]
    T = _line(n, w)
    x, psd = _strain(n)
    rows = _rows(T, n // 2, 3)
    d = api.make_desc(2048.0, n, 1, T, w=w, rho_ii=0.0)  # a trigger from every window
    room = T * n // (2 * w)

    def call():
        buf, nt = api.rb_filter_plain(d, rows, x, psd, capacity=room)
        assert nt == room
        rec = buf.view(torch.int64).view(-1, 3)[:nt]
        sample, tmpl = rec[:, 0], rec[:, 1] & 0xFFFFFFFF
        order = torch.sort(tmpl * n + sample)[1]
        return sample[order] // w + tmpl[order] * n, sample[order], rec.view(torch.float32).view(-1, 6)[order, 4]

    ((win, m, snr), one), ((win0, m0, snr0), two) = _both(env, call)
    assert one < two
    assert torch.equal(win, win0)
    assert (snr - snr0).abs().max() <= 2 * TOL * snr0.square().mean().sqrt()
    assert (m != m0).sum() <= 1e-4 * len(m)  # (only between samples that are equal to rounding)


# blocks have at most 2^20 samples
@pytest.mark.parametrize("m,w,lowpass", [(m, w, lowpass) for m in LENGTHS[:6] for w, lowpass in ((2, False), (8, False), (2, True))
                                         if m * w <= 1 << 20])
@pytest.mark.parametrize("above", [True, False])
def test_folded_stage(env, m, w, lowpass, above):
    api = env[0]
    n, T = m * w, _fold_line(m, lowpass) - (not above)
    x, psd = _strain(n)
    rows = _rows(T, n // 2, 4)
    room = T * m // 2
    d = api.make_desc(2048.0, n, 1, T, w=w, rho_i=0.0, cand_capacity=room)  # a candidate from every bin

    def call():
        buf, nc = (api.rb_stage1_lowpass if lowpass else api.rb_stage1_folded)(d, rows, x, psd)
        assert nc == room
        rec = buf.view(torch.int32).view(-1, 4)[:nc]
        key = rec[:, 0].long() * m + rec[:, 1]
        order = torch.sort(key)[1]
        return key[order], rec.view(torch.float32)[order, 2]

    ((key, snr), _), ((key0, snr0), _) = _both(env, call)
    assert torch.equal(key, key0)
    # (two paths do not give the same last bits)
    assert torch.equal(snr, snr0) == (not above or (lowpass and m < 1 << 19))
    assert (snr - snr0).abs().max() <= 2 * TOL * snr0.square().mean().sqrt()
