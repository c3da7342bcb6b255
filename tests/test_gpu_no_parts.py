"""A system whose allocator has no room for the parts of its convolution streams
whole rings: the same bits, alone and as one member of a batch (needs a GPU)."""
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


def _system(n, m_max, refuse, monkeypatch, **kw):
    """With refuse, the second allocation of set_kernels (the first is the radial table) fails."""
    from paper_1808_00270_gb300 import GLD, binding, inputs

    class Allocator(binding._TorchAllocator):
        def __init__(self):
            super().__init__()
            self.inner, self.asked = self.alloc, None

            def alloc(nbytes, stream, user):
                if self.asked is not None:
                    self.asked += 1
                    if self.asked == 2:
                        return None
                return self.inner(nbytes, stream, user)
            self.alloc = binding.ALLOC_FN(alloc)

    w = inputs.Workload("np", n=n, box=inputs.box_for_density(n, 0.1), m_max=m_max, dt=0.005, r_c=2.0, tau_s=0.5,
                        tau_p=0.3, steps=1, seed=9)
    pos, vel = inputs.initial_state(w)
    with monkeypatch.context() as mp:
        mp.setattr(binding, "_TorchAllocator", Allocator)
        g = GLD(n=n, box=w.box, dt=w.dt, m_max=m_max, r_c=w.r_c, A_cons=w.A_cons, pos=pos, vel=vel, seed=w.seed, **kw)
    before = g.bytes()
    g._alloc.asked = 0 if refuse else None
    ks, gk, f, dr = kernels(w)
    g.set_kernels(ks, g=gk, f=f, dr=dr)
    assert refuse == (g.bytes() - before < 16 * 2 * 12 * n)  # two accumulators, at least 16 rows of parts
    g._alloc.asked = None
    return g


def _result(g):
    from paper_1808_00270_gb300 import ARR_DISP, ARR_FC, ARR_FD, ARR_FR, ARR_HIST
    return [*g.get_state()] + [g.get(k) for k in (ARR_DISP, ARR_FC, ARR_FD, ARR_FR, ARR_HIST)]


# four ranges of slots, in FP32 and BF16; steps in a cluster and step kernels;
# past the cluster kernel
@pytest.mark.parametrize("n,m_max,kw", [(300, 100, {}), (1000, 131, dict(hist_dtype="bf16")), (6000, 70, {}), (500, 70, dict(kahan=True))])
def test_alone(n, m_max, kw, monkeypatch):
    got = []
    for graphs, refuse in ((1, True), (2, True), (0, True), (1, False)):
        g = _system(n, m_max, refuse, monkeypatch, use_graphs=graphs, **kw)
        for k in (64, 1, 7, 70, 18):
            g.step(k)
        got.append(_result(g))
        g.close()
    for other in got[1:]:
        for x, y in zip(got[0], other):
            assert np.array_equal(x, y)


def test_in_a_batch(monkeypatch):
    from paper_1808_00270_gb300 import Batch
    got = []
    for refuse in ((False, False, False), (False, True, False)):
        ms = [_system(n, m, r, monkeypatch) for (n, m), r in zip(((300, 100), (700, 70), (5000, 66)), refuse)]
        b = Batch()
        for g in ms:
            b.add(g)
        for k in (64, 128, 64):
            b.step(k)
        b.sync()
        got.append([x for g in ms for x in _result(g)])
    for x, y in zip(*got):
        assert np.array_equal(x, y)
