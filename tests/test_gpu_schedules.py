"""The convolution schedules of a batch (needs a GPU)."""
import pytest

from gld_cases import make_gpu

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.set_device(0)


def test_schedules_are_timed_on_whole_rings():
    """What a schedule is timed on does not depend on the members' place in their
    rings: at step 0, and where a step of a block streams 16 of 399 rows."""
    from paper_1808_00270_gb300 import Batch, inputs
    w = inputs.Workload("sched", n=60000, box=inputs.box_for_density(60000, 0.05), m_max=400, dt=0.005, r_c=2.0,
                        tau_s=0.5, tau_p=0.3, steps=1, seed=6)
    g = make_gpu(w)
    times = []
    for steps in (384, 64):
        b = Batch()
        b.add(g)
        b.step(steps)
        b.sync()
        times.append(min(b.info()["schedule_ms"][:3]))
        b.remove(g)
        b.close()
    assert 0.5 < times[1] / times[0] < 2.0, times
    g.close()
