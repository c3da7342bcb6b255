"""Small systems step inside one kernel (a thread-block cluster); use_graphs=2
keeps the launches of the step kernels.  Both give the same bits, for sizes at
the edges of the kernel's lanes and CTAs and for every option it takes (needs a
GPU)."""
import numpy as np
import pytest

from gld_cases import kernels

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.set_device(0)


def _system(w, graphs, pair=True, table=False, **kw):
    from paper_1808_00270_gb300 import GLD, inputs
    pos, vel = inputs.initial_state(w)
    g = GLD(n=w.n, box=w.box, dt=w.dt, m_max=w.m_max, r_c=w.r_c, A_cons=w.A_cons, pos=pos, vel=vel, seed=w.seed,
            use_graphs=graphs, vacf_len=60, vacf_stride=4, vacf_burnin=3, **kw)
    ks, gk, f, dr = kernels(w)
    g.set_kernels(ks, g=gk, f=f, dr=dr) if pair else g.set_kernels(ks)
    if table:
        r = np.linspace(0.0, w.r_c, 200)
        g.set_conservative_table(10.0 * (1 - r / w.r_c), dr=r[1])
    return g


def _result(g):
    from paper_1808_00270_gb300 import ARR_DISP, ARR_FC, ARR_FD, ARR_FR, ARR_HIST
    p, v = g.get_state()
    c, n = g.vacf()
    return [p, v, c, np.array([n, g.step_index, g.diag()["rebuilds"]])] + [
        g.get(k) for k in (ARR_DISP, ARR_FC, ARR_FD, ARR_FR, ARR_HIST)]


# one particle; 8 lanes: one CTA and its edge, 16 CTAs full; 4 lanes and 2 lanes
# and their edges; one cell (a box below three list radii); dense boxes
@pytest.mark.parametrize("n,rho,m_max,kw", [
    (1, 0.001, 2, {}), (2, 0.02, 33, {}), (64, 0.125, 32, {}), (65, 0.5, 40, {}), (64, 0.1, 64, dict(pair=False)),
    (300, 0.05, 100, dict(hist_dtype="bf16")), (1024, 0.1, 130, {}), (1025, 0.1, 70, dict(table=True)),
    (2048, 0.2, 100, dict(hist_dtype="bf16", pair=False)), (2049, 0.02, 65, {}), (4096, 0.1, 200, {})])
def test_same_bits_as_the_step_kernels(n, rho, m_max, kw):
    from paper_1808_00270_gb300 import inputs
    short = m_max < 58
    w = inputs.Workload("cl", n=n, box=max(inputs.box_for_density(n, rho), 4.5), m_max=m_max, dt=0.01 if short else 0.005,
                        r_c=2.0, tau_s=0.2 if short else 0.5, tau_p=0.1 if short else 0.3, steps=1, seed=n)
    psd = dict(psd_clamp=True) if m_max < 17 else {}
    a, b = _system(w, 1, **kw, **psd), _system(w, 2, **kw, **psd)
    for k in (64, 1, 7, 70, 18):  # graph blocks, parts of blocks, block starts off the multiples of 16
        a.step(k)
    b.step(160)
    assert a.diag()["graph_mode"] == 1
    for x, y in zip(_result(a), _result(b)):
        assert np.array_equal(x, y)
    a.step(64)
    b.step(64)
    for x, y in zip(_result(a), _result(b)):
        assert np.array_equal(x, y)
    a.close()
    b.close()


@pytest.mark.parametrize("n,rho", [(64, 0.5), (12288, 0.1), (12289, 0.1), (40000, 0.3)])
def test_lists_hold_every_pair_after_rebuilds(n, rho):
    """Lists built by a cluster and by lanes over cell rows, after steps with
    rebuilds: the pairs are the brute-force pairs of the same positions."""
    import oracle
    from paper_1808_00270_gb300 import inputs
    w = inputs.Workload("nb", n=n, box=max(inputs.box_for_density(n, rho), 4.5), m_max=64, dt=0.005, r_c=2.0, tau_s=0.5,
                        tau_p=0.3, steps=1, seed=n)
    g = _system(w, 1)
    g.step(40)
    assert g.diag()["rebuilds"] > 2
    p, _ = g.get_state()
    got = {tuple(x) for x in g.pairs().tolist()}
    want = {tuple(x) for x in oracle.pairs_brute_f32(p.astype(np.float32), w.box, np.float32(w.r_c ** 2)).tolist()}
    assert got == want
    g.close()
