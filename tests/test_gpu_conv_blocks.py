"""The history convolution over blocks of steps (needs a GPU): a step whose
sums are resumed from its block's parts gives the bits of the whole sum over
the ring, wherever the rewritten slots lie in the ring and in its split into
ranges."""
import numpy as np
import pytest

from gld_cases import make_gpu

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.set_device(0)


def _whole_sums(g, w, hist, coef, step, bf16, kahan):
    """hist_conv_dev over the ring that `hist` (entry m - 1: dR_{step-m}) stands for."""
    from paper_1808_00270_gb300 import hist_conv_dev
    H, n_pad, order = w.m_max - 1, (w.n + 31) // 32 * 32, g.order()
    ring = np.zeros((H, 3, n_pad), dtype=np.float32)
    for m in range(1, H + 1):
        ring[(step - m) % H, :, : w.n] = hist[m - 1][order].T
    d_ring = torch.from_numpy(ring).cuda()
    if bf16:
        d_ring = d_ring.to(torch.bfloat16)
    nacc = coef.shape[0]
    out = torch.zeros((nacc, 3, n_pad), dtype=torch.float32, device="cuda")
    hist_conv_dev(d_ring, n_pad, w.m_max, step, torch.from_numpy(coef).cuda(), nacc, out, bf16=bf16, kahan=kahan)
    torch.cuda.synchronize()
    got = np.empty((nacc, w.n, 3), dtype=np.float32)
    got[:, order] = out.cpu().numpy()[:, :, : w.n].transpose(0, 2, 1)
    return got


# shortest ring with blocks (32 slots), a split into four ranges, odd sizes, one
# range (columns that fill the chip), three accumulators, BF16, compensated sums
# (columns of 4, 8 and 16 bytes)
@pytest.mark.parametrize("n,m_max,terms,hist,kahan", [
    (64, 33, "pair", "f32", False), (77, 34, "pair", "f32", False), (1001, 100, "pair", "f32", False),
    (1001, 131, "general", "f32", False), (1001, 100, "pair", "bf16", False), (1001, 100, "pair", "f32", True),
    (333, 70, "general", "bf16", True), (90001, 66, "pair", "f32", False), (90001, 66, "pair", "bf16", True),
    (120001, 40, "pair", "bf16", True), (160001, 40, "pair", "bf16", True)])
def test_resumed_sums_are_the_whole_sums(n, m_max, terms, hist, kahan):
    from paper_1808_00270_gb300 import ARR_CONV, ARR_HIST, inputs
    short = m_max < 58
    w = inputs.Workload("blk", n=n, box=inputs.box_for_density(n, 0.1), m_max=m_max, dt=0.01 if short else 0.005,
                        r_c=2.0, tau_s=0.2 if short else 0.5, tau_p=0.1 if short else 0.3, steps=1, seed=3)
    ks = inputs.self_kernel_samples(w)
    gk, f, dr = inputs.pair_kernel_tables(w)
    g = make_gpu(w, hist_dtype=hist, kahan=kahan)
    rows = [ks, gk[0]]
    if terms == "general":
        g.set_kernels(ks, g=gk, f=f, dr=dr, gs=0.5 * gk, fs=0.3 * f)
        rows.append(0.5 * gk[0])
    coef = np.stack([np.asarray(r) * w.dt * np.where(np.arange(m_max) == 0, 0.5, 1.0) for r in rows]).astype(np.float32)
    g.step(64)
    # numbers in a block, block starts, and the wrap of the ring
    at = (64, 65, 71, 72, 79, 80, 95, 96, 101, 127, 128, 130)
    for step in at if n < 50000 else at[:6]:
        g.step(step - g.step_index)
        h = g.get(ARR_HIST)
        g.step(1)
        got = g.get(ARR_CONV).astype(np.float32)
        assert np.array_equal(got, _whole_sums(g, w, h, coef, step, hist == "bf16", kahan)), step
    g.close()
