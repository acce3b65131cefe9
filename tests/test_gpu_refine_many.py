"""More candidates than CTAs of one launch: the ascent takes two CTAs each, and a grid holds less than 2^31."""
import pytest

from paper_2110_13115_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_more_candidates_than_a_launch_holds():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2110_13115_gb300 import _native as N, api

    count = (1 << 30) + 1
    if torch.cuda.mem_get_info()[0] < count * 80 + (1 << 32):
        pytest.skip("needs 84 GB")
    n = 1 << 10
    psd = torch.from_numpy(inputs.analytic_psd(inputs.Grid(2048.0, n, 30.0))).cuda()
    s_hat = torch.ones(n // 2, dtype=torch.complex64, device="cuda")
    theta = torch.zeros((count, 4), dtype=torch.float64, device="cuda")  # refused one by one, which takes no time
    try:
        with pytest.raises(N.RBError, match="eta outside") as e:
            api.rb_refine(api.make_refine_desc(2048.0, n, 30.0, steps=1), s_hat, psd, theta)
        assert e.value.code == N.RB_ERR_BAD_INPUT
    finally:
        del theta
        torch.cuda.empty_cache()
