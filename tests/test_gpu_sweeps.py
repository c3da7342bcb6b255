"""Where the sweeps of the pair noise run in one launch, and one launch with more
pairs than a thread keeps (needs a GPU)."""
import pytest

from gld_cases import rel_l2
from test_gpu_lanes import _system

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.set_device(0)


def _launches(g, degree):
    n = g.profile_steps(64)["pair_noise"][1] // 64
    assert n in (1, degree)
    return n


# blocks of 128 threads per SM (on 152): two and three, four, five, six; degrees on
# both sides of the line; mean pairs inside the cutoff against the room for them
@pytest.mark.parametrize("n,rho,degree,one", [
    (38912, 0.05, 2, True), (58368, 0.05, 2, True), (58369, 0.05, 2, False), (77824, 0.05, 3, True),
    (77825, 0.05, 3, False), (97280, 0.05, 4, True), (97281, 0.05, 8, False),
    (60000, 0.50, 4, True), (60000, 0.52, 4, False)])
def test_where_one_launch_takes_all_sweeps(n, rho, degree, one):
    g = _system(n, rho, degree=degree)
    assert (_launches(g, degree) == 1) == one
    g.close()


def test_more_pairs_than_a_thread_keeps():
    """17 pairs on average and room for 20: against a launch per sweep (a vanishing
    perpendicular factor), which adds nothing but roundings, at most 2 K (pairs + 4)
    of 6e-8 each, adding up at random."""
    from paper_1808_00270_gb300 import ARR_FR
    a, b = _system(60000, 0.50, degree=4), _system(60000, 0.50, degree=4, perp0=True)
    a.step(1)
    b.step(1)
    assert rel_l2(a.get(ARR_FR), b.get(ARR_FR)) < 1e-5
    assert _launches(a, 4) == 1 and _launches(b, 4) == 4
    a.close()
    b.close()
