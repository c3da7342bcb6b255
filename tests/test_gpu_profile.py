"""gld_profile_steps counts the kernels it launches (needs a GPU)."""
import pytest

from gld_cases import kernels, make_gpu

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.set_device(0)


def _workload(n, m_max):
    from paper_1808_00270_gb300 import inputs
    return inputs.Workload("prof", n=n, box=inputs.box_for_density(n, 0.05), m_max=m_max, dt=0.005, r_c=2.0, tau_s=0.5,
                           tau_p=0.3, steps=1, seed=3)


# blocks of 8 steps (a split into ranges) and of 16, memories too short for
# blocks; lists built by one kernel and by four
@pytest.mark.parametrize("n,m_max,block,lists", [(4097, 200, 8, 1), (8193, 170, 8, 4), (150001, 66, 16, 4), (5000, 100, 0, 1), (5000, 32, 0, 1)])
def test_launches_of_a_step(n, m_max, block, lists):
    g = make_gpu(_workload(n, m_max), psd_clamp=True)
    d = g.diag()
    assert d["conv_block"] == block and (block == 0 or (d["conv_ranges"] > 1) == (block == 8))
    p = g.profile_steps(128)
    assert p["hist_conv"][1] == 128 + (128 // block if block else 0)
    assert p["cell_build"][1] == 128 * lists
    assert p["pair_force_integrate"][1] == p["cforce"][1] == 128 and p["noise"][1] == 2 * 2
    g.close()


def test_launches_of_three_accumulators():
    w = _workload(4097, 200)
    g = make_gpu(w)
    ks, gk, f, dr = kernels(w)
    g.set_kernels(ks, g=gk, f=f, dr=dr, gs=0.5 * gk, fs=0.3 * f)
    assert g.profile_steps(64)["hist_conv"][1] == 64 + 2 * 8
    g.close()


@pytest.mark.parametrize("perp,sweeps", [(False, 1), (True, 4)])
def test_launches_of_the_sweeps(perp, sweeps):
    """One cooperative launch for all sweeps, or one each with perpendicular factors."""
    w = _workload(3000, 200)
    g = make_gpu(w)
    ks, gk, f, dr = kernels(w)
    g.set_kernels(ks, g=gk, f=0.1 * f, dr=dr)
    if perp:
        g.set_perpendicular(fp=1e-12 * f)
    g.set_pair_noise(4, lam=2.0)
    p = g.profile_steps(64)
    name = [k for k in p if "noise" in k and k != "noise"][0]
    assert p[name][1] == 64 * sweeps and p["noise"][1] == 2 + 4
    g.close()
