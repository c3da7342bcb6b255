"""Neighbour lists against all pairs at the last size that a cluster builds, the
last that lanes over the grid build alone, and one past each (needs a GPU)."""
import numpy as np
import pytest

import oracle
from gld_cases import make_gpu

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.set_device(0)


@pytest.mark.parametrize("n,kernels", [(8192, 1), (8193, 4), (65536, 4), (65537, 4)])
def test_lists_hold_every_pair_after_rebuilds(n, kernels):
    from paper_1808_00270_gb300 import inputs
    w = inputs.Workload("edge", n=n, box=inputs.box_for_density(n, 0.1), m_max=40, dt=0.01, r_c=2.0, tau_s=0.2, tau_p=0.1,
                        steps=1, seed=n)
    g = make_gpu(w)
    g.step(40)
    assert g.diag()["rebuilds"] > 2
    p, _ = g.get_state()
    got = {tuple(x) for x in g.pairs().tolist()}
    want = {tuple(x) for x in oracle.pairs_brute_f32(p.astype(np.float32), w.box, np.float32(w.r_c ** 2)).tolist()}
    assert got == want
    assert g.profile_steps(64)["cell_build"][1] == 64 * kernels
    g.close()
