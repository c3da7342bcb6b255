"""The shortest memories whose convolution a system alone forms in blocks of steps,
and one slot less (needs a GPU)."""
import pytest

import test_gpu_conv_blocks
from gld_cases import make_gpu

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.set_device(0)


# four ranges of few, more and many columns; two; one (a wave, below more); BF16; compensated sums of
# few and many columns
LINES = [(5000, 192, "f32", False), (8193, 144, "f32", False), (40001, 96, "f32", False), (90001, 56, "f32", False), (150001, 32, "f32", False),
         (12001, 144, "bf16", False), (140001, 96, "bf16", False),
         (5000, 96, "f32", True), (30001, 160, "f32", True), (120001, 64, "f32", True), (12001, 96, "bf16", True), (100001, 192, "bf16", True)]


@pytest.mark.parametrize("n,slots,hist,kahan", LINES)
def test_resumed_sums_at_the_line(n, slots, hist, kahan):
    test_gpu_conv_blocks.test_resumed_sums_are_the_whole_sums(n, slots + 1, "pair", hist, kahan)


@pytest.mark.parametrize("n,slots,hist,kahan", LINES + [(600001, 56, "f32", False), (600001, 56, "bf16", False), (300001, 4000, "bf16", True)])
def test_where_blocks_begin(n, slots, hist, kahan):
    from paper_1808_00270_gb300 import inputs
    never = slots == 4000
    for m_max in ((201,) if never else (slots, slots + 1)):
        short = m_max < 58
        w = inputs.Workload("rule", n=n, box=inputs.box_for_density(n, 0.1), m_max=m_max, dt=0.01 if short else 0.005,
                            r_c=2.0, tau_s=0.2 if short else 0.5, tau_p=0.1 if short else 0.3, steps=1, seed=3)
        g = make_gpu(w, hist_dtype=hist, kahan=kahan)
        assert (g.diag()["conv_block"] > 0) == (not never and m_max > slots)
        g.close()
