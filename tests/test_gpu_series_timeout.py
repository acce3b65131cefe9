"""Failure detection of the fused transforms: their waits are bounded (2 s of %globaltimer). A host-only test hook makes the
next launch's second part wait for a count that nothing reaches; the wait runs out, the launch stops and returns.
Calls that read the status report RB_ERR_TIMEOUT, the basis filter, which only enqueues, leaves NaN in every value, and
the next call on the same workspace is right."""
import time

import numpy as np
import pytest

from paper_2110_13115_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def block():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2110_13115_gb300 import _native as N, api

    n, rows, w = 1 << 15, 512, 2  # 2^24 points; folded 2^23
    grid = inputs.Grid(2048.0, n, 30.0)
    psd = inputs.analytic_psd(grid)
    x = torch.from_numpy(inputs.coloured_noise(grid, psd, 4).astype(np.float32)).cuda()
    p = torch.from_numpy(inputs.unit_rows(rows, n // 2, 6).astype(np.complex64)).cuda()
    lib = N.load()
    yield api, N, lib, n, rows, w, torch.from_numpy(psd).cuda(), x, p
    lib.rbx_series_withhold(0)


def _basis_call(block):
    api, N, lib, n, rows, w, psd, x, p = block
    d = api.make_desc(2048.0, n, rows, 1, w=w)
    basis = api.Basis(p, torch.ones((1, rows), dtype=torch.complex64, device="cuda"), n)
    ws = api.workspace(d)
    return d, basis, api.rb_whiten(d, x, psd, ws=ws), ws


@pytest.mark.parametrize("keep_beta", [True, False])
def test_basis_filter_leaves_nan(block, keep_beta):
    api, N, lib = block[:3]
    d, basis, sh, ws = _basis_call(block)
    beta, bavg = api.rb_basis_filter(d, basis, sh, ws=ws)
    assert torch.isfinite(torch.view_as_real(beta)).all()
    lib.rbx_series_withhold(1)
    t0 = time.perf_counter()
    bad, bad_avg = api.rb_basis_filter(d, basis, sh, keep_beta=keep_beta, ws=ws)
    torch.cuda.synchronize()
    assert 1.0 < time.perf_counter() - t0 < 30.0
    assert torch.isnan(torch.view_as_real(bad_avg)).all()
    assert bad is None if not keep_beta else torch.isnan(torch.view_as_real(bad)).all()
    again, again_avg = api.rb_basis_filter(d, basis, sh, ws=ws)
    assert torch.equal(again, beta) and torch.equal(again_avg, bavg)


def _timed_out(block, call):
    N, lib = block[1:3]
    want = call()
    lib.rbx_series_withhold(1)
    with pytest.raises(N.RBError) as e:
        call()
    assert e.value.code == N.RB_ERR_TIMEOUT and b"timed out" in lib.rb_last_error_detail()
    torch.cuda.synchronize()
    assert call() == want


def test_template_method_reports(block):
    api, N, lib, n, rows, w, psd, x, p = block
    d = api.make_desc(2048.0, n, 1, rows, w=w, rho_ii=3.5)
    _timed_out(block, lambda: api.rb_filter_plain(d, p, x, psd)[1])


def test_folded_stage_reports(block):
    api, N, lib, n, rows, w, psd, x, p = block
    d = api.make_desc(2048.0, n, 1, rows, w=w, rho_i=3.5, cand_capacity=1 << 20)
    _timed_out(block, lambda: api.rb_stage1_folded(d, p, x, psd)[1])


def test_tuner_reports(block):
    api = block[0]
    d, basis, sh, ws = _basis_call(block)
    _timed_out(block, lambda: api.rb_tune_fft(d, basis, sh, ws=ws)[0])
