"""The three forms of use_graphs take the kernels they name and give the same
bits (needs a GPU)."""
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


def _three_forms(n, m_max, calls):
    from paper_1808_00270_gb300 import ARR_DISP, ARR_FC, ARR_FD, ARR_FR, ARR_HIST, inputs
    w = inputs.Workload("form", n=n, box=inputs.box_for_density(n, 0.1), m_max=m_max, dt=0.01, r_c=2.0, tau_s=0.2,
                        tau_p=0.1, steps=1, seed=7)
    diag, got = [], []
    for form in (0, 1, 2):
        g = make_gpu(w, use_graphs=form)
        for k in calls:
            g.step(k)
        diag.append(g.diag())
        got.append([*g.get_state()] + [g.get(a) for a in (ARR_DISP, ARR_FC, ARR_FD, ARR_FR, ARR_HIST)])
        g.close()
    for other in got[1:]:
        for x, y in zip(got[0], other):
            assert np.array_equal(x, y)
    assert len({d["rebuilds"] for d in diag}) == 1 and diag[0]["rebuilds"] > 1
    return diag


@pytest.mark.parametrize("n", [64, 300, 4096])
def test_small_systems(n):
    """use_graphs = 0 and 2 launch the step kernels; 1 steps inside a kernel."""
    d0, d1, d2 = _three_forms(n, 40, [64, 1, 7, 70, 18])
    assert d0["graph_mode"] == 0 and d0["cluster_steps"] == 0 and d2["cluster_steps"] == 0
    assert d1["cluster_steps"] > 0 and d2["graph_mode"] == 1


def test_rebuild_in_a_conditional_node():
    """Blocks, single steps until pieces of a block are replayed, pieces, a block."""
    d0, d1, d2 = _three_forms(262144, 40, [64, 64] + [1] * 70 + [10, 32, 16, 64])
    assert (d0["graph_mode"], d1["graph_mode"], d2["graph_mode"]) == (0, 2, 1)
