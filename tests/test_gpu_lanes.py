"""Lanes per particle, the sweeps of the pair noise in one launch and the
replayed segments of single steps against the tile kernels of a batch, a launch
per sweep and blocks of steps (needs a GPU)."""
import numpy as np
import pytest

from gld_cases import kernels, rel_l2

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.set_device(0)


def _system(n, rho, terms="pair", degree=0, vacf=0, kT=1.0, perp0=False, seed=11):
    from paper_1808_00270_gb300 import GLD, inputs
    w = inputs.Workload("lanes", n=n, box=max(inputs.box_for_density(n, rho), 4.5), m_max=200 if degree else 66,
                        dt=0.005, r_c=2.0, tau_s=0.5, tau_p=0.3, steps=1, seed=seed)
    pos, vel = inputs.initial_state(w)
    g = GLD(n=n, box=w.box, dt=w.dt, m_max=w.m_max, r_c=w.r_c, A_cons=w.A_cons, pos=pos, vel=vel, seed=seed, kT=kT,
            kahan=True, vacf_len=vacf, vacf_stride=4, vacf_burnin=1)
    ks, gk, f, dr = kernels(w)
    if degree:
        f = 0.1 * min(1.0, 0.05 / rho) * f  # rows of the pair matrix below its bound
    if terms == "general":
        g.set_kernels(ks, g=gk, f=f, dr=dr, gs=0.5 * gk, fs=0.3 * f)
        g.set_perpendicular(fp=0.4 * f, fs=0.1 * f)
    else:
        g.set_kernels(ks, g=gk, f=f, dr=dr)
    if perp0:
        g.set_perpendicular(fp=1e-12 * f)
    if degree:
        g.set_pair_noise(degree, lam=2.0)
    return g


def _same(a, b):
    from paper_1808_00270_gb300 import ARR_DISP, ARR_FC, ARR_FD, ARR_FR, ARR_HIST
    for k in (ARR_DISP, ARR_FC, ARR_FD, ARR_FR, ARR_HIST):
        assert np.array_equal(a.get(k), b.get(k))
    for x, y in zip(a.get_state(), b.get_state()):
        assert np.array_equal(x, y)
    assert a.diag()["rebuilds"] == b.diag()["rebuilds"] > 0


# past the cluster kernel; eight lanes to four, four to one; lists built by lanes
# in a cluster, over the grid (both ends) and by one thread per particle
@pytest.mark.parametrize("n,terms,vacf", [
    (4097, "pair", 0), (8193, "pair", 40), (19456, "general", 0), (19457, "general", 40), (19457, "pair", 0),
    (22528, "pair", 40), (22529, "general", 0), (65536, "pair", 0), (65537, "pair", 0)])
def test_lanes_give_the_bits_of_the_tile_kernels(n, terms, vacf):
    """At kT = 0 (the filters of a system alone and in a batch round differently)
    and with compensated sums (one range of slots in both): nothing else differs."""
    from paper_1808_00270_gb300 import Batch
    alone, member = (_system(n, 0.1, terms, vacf=vacf, kT=0.0) for _ in range(2))
    b = Batch()
    b.add(member)
    alone.step(128)
    b.step(128)
    b.sync()
    _same(alone, member)
    alone.close()
    member.close()


# one block and a ragged last one, two to eight sweeps, more pairs per particle
# than a thread keeps.  One step; a vanishing perpendicular factor takes a launch
# per sweep and adds nothing but roundings: at most 2 K (pairs + 4) of 6e-8 each,
# which add up at random.
@pytest.mark.parametrize("n,rho,degree", [(100, 0.05, 2), (129, 0.05, 8), (3000, 0.05, 3), (20001, 0.3, 4), (60000, 1.0, 4)])
def test_sweeps_of_one_launch_match_a_launch_each(n, rho, degree):
    from paper_1808_00270_gb300 import ARR_FR
    a, b = _system(n, rho, degree=degree), _system(n, rho, degree=degree, perp0=True)
    a.step(1)
    b.step(1)
    assert rel_l2(a.get(ARR_FR), b.get(ARR_FR)) < 1e-5
    a.close()
    b.close()


@pytest.mark.parametrize("n,degree", [(5000, 0), (24001, 0), (3000, 4)])
def test_single_steps_give_the_bits_of_blocks(n, degree):
    """More single steps than run eagerly, then replayed segments, off the blocks' boundaries."""
    a, b = _system(n, 0.05, degree=degree), _system(n, 0.05, degree=degree)
    for k in [1] * 150 + [7, 3, 32]:
        a.step(k)
    b.step(192)
    _same(a, b)
    a.close()
    b.close()
