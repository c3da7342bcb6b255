"""Dense systems of more particles than the cluster has lanes to spare step by the
step kernels; the same bits (needs a GPU)."""
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


# (4/3 pi 2.4^3 entries per unit of density) eight lanes: any list; four: up to 24;
# two: up to 8
@pytest.mark.parametrize("n,rho,cluster", [(1024, 0.8, True), (1025, 0.41, True), (1025, 0.42, False), (2048, 0.42, False),
                                           (2049, 0.13, True), (2049, 0.145, False), (4096, 0.8, False)])
def test_long_lists_leave_the_cluster(n, rho, cluster):
    from paper_1808_00270_gb300 import inputs
    w = inputs.Workload("dense", n=n, box=inputs.box_for_density(n, rho), m_max=70, dt=0.005, r_c=2.0, tau_s=0.5,
                        tau_p=0.3, steps=1, seed=7)
    a, b = make_gpu(w, use_graphs=1), make_gpu(w, use_graphs=0)
    for k in (1, 7, 30, 64, 3):
        a.step(k)
    b.step(105)
    assert (a.diag()["cluster_steps"] > 0) == cluster and b.diag()["cluster_steps"] == 0
    for x, y in zip(a.get_state(), b.get_state()):
        assert np.array_equal(x, y)
    a.close()
    b.close()
