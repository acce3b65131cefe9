"""The FFT tuner chooses among schedules that differ: rows that take the fused launch have one, and tuning on them leaves
the choice for the two passes of few rows of the same length and width alone."""
import pytest

from paper_2110_13115_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

PINNED = 5  # the intermediate's chunks hold 128 rows of 2^16 samples, those of the variant 0 half as many


def test_tuning_of_the_fused_launch_leaves_the_passes_alone():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2110_13115_gb300 import _native as N, api

    n, w, k = 1 << 16, 8, 128  # 2^23 points: the fused launch; one row fewer takes the passes
    rows = torch.from_numpy(inputs.unit_rows(k, n // 2, seed=3).astype("complex64")).cuda()
    one = torch.ones((1, k), dtype=torch.complex64, device="cuda")
    sh = torch.view_as_complex(torch.randn((n // 2, 2), device="cuda"))

    def launches(count):
        d = api.make_desc(2048.0, n, count, 1, w=w)
        basis = api.Basis(rows[:count], one[:, :count].contiguous(), n)
        before = api.rb_kernel_launches()
        api.rb_basis_filter(d, basis, sh)
        return api.rb_kernel_launches() - before - 1  # (the tables)

    d = api.make_desc(2048.0, n, k, 1, w=w)
    try:
        assert launches(k) == 1 and launches(k - 1) == 4
        api.rb_set_fft_variant(d, PINNED)
        assert launches(k) == 1 and launches(k - 1) == 2
        chosen, times = api.rb_tune_fft(d, api.Basis(rows, one, n), sh)
        assert chosen == 0 and len(set(times)) == 1 and times[0] > 0
        assert launches(k - 1) == 2
        # few rows: every schedule is timed, and the fastest is taken
        few = api.make_desc(2048.0, n, 20, 1, w=w)
        chosen, times = api.rb_tune_fft(few, api.Basis(rows[:20], one[:, :20].contiguous(), n), sh)
        assert times[chosen] == min(times) and len(set(times)) > 1 and len(times) == N.RB_FFT_VARIANTS
    finally:
        api.rb_set_fft_variant(d, 0)
