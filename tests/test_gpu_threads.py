"""Systems of several host threads and streams do not get in each other's way: the
dynamic shared memory allowed per function, and grids that wait for all of their
blocks (needs a GPU)."""
import threading

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


def test_a_shorter_memory_leaves_a_longer_one_its_shared_memory():
    """147 KB of weights, then 72 KB of another length, then the first again."""
    from paper_1808_00270_gb300 import hist_conv_dev
    n_pad, nacc, got = 64, 9, []
    for m_max in (4096, 2000, 4096):
        rng = np.random.default_rng(m_max)
        ring = torch.from_numpy(rng.standard_normal((m_max - 1, 3, n_pad)).astype(np.float32)).cuda()
        coef = torch.from_numpy(rng.standard_normal((nacc, m_max)).astype(np.float32)).cuda()
        out = torch.zeros((nacc, 3, n_pad), dtype=torch.float32, device="cuda")
        hist_conv_dev(ring, n_pad, m_max, 7, coef, nacc, out)
        torch.cuda.synchronize()
        got.append(out.cpu().numpy())
    assert np.array_equal(got[0], got[2])


# (steps in one cluster; list builds in a cluster and step kernels of their own)
@pytest.mark.parametrize("sizes", [((300, 0.05, 40), (500, 0.3, 400)), ((4500, 0.05, 40), (4600, 0.3, 400))])
def test_two_threads_step_systems_of_their_own(sizes):
    """Single steps from two host threads, each on its own stream and system:
    the results of one thread after the other."""
    from paper_1808_00270_gb300 import GLD, inputs
    ws = [inputs.Workload("t%d" % k, n=n, box=inputs.box_for_density(n, rho), m_max=m, dt=0.01 if m < 58 else 0.005,
                          r_c=2.0, tau_s=0.2 if m < 58 else 0.5, tau_p=0.1 if m < 58 else 0.3, steps=1, seed=3 + k)
          for k, (n, rho, m) in enumerate(sizes)]
    errors, out = [], {}

    def work(key, w, steps):
        try:
            torch.cuda.set_device(0)
            with torch.cuda.stream(torch.cuda.Stream()):
                for rep in range(3):  # creation and kernels race too
                    g = make_gpu(w, torch_allocator=False)
                    for _ in range(steps):
                        g.step(1)
                    out[key, rep] = g.get_state()
                    g.close()
        except Exception as e:  # noqa: BLE001
            errors.append(repr(e))

    for k, w in enumerate(ws):
        work(("alone", k), w, 700)
    assert not errors
    threads = [threading.Thread(target=work, args=(("both", k), w, 700)) for k, w in enumerate(ws)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
    for k in range(2):
        for rep in range(3):
            for x, y in zip(out[("alone", k), 0], out[("both", k), rep]):
                assert np.array_equal(x, y)


def test_two_threads_with_pair_noise():
    """The sweeps are one launch whose blocks wait for each other (a bounded wait),
    and each system's fill the chip: two of them, on streams of their own, one
    step and one wait at a time, give the results of one after the other."""
    from paper_1808_00270_gb300 import GLD, inputs
    w = inputs.Workload("pn", n=32768, box=inputs.box_for_density(32768, 0.05), m_max=128, dt=0.005, r_c=2.0, tau_s=0.5,
                        tau_p=0.3, steps=1, seed=5)
    errors, out = [], {}

    def work(key):
        try:
            torch.cuda.set_device(0)
            with torch.cuda.stream(torch.cuda.Stream()):
                g = make_gpu(w, torch_allocator=False, pair=False)
                gk, f, dr = inputs.pair_kernel_tables(w)
                g.set_kernels(inputs.self_kernel_samples(w), g=gk, f=0.2 * f, dr=dr)
                g.set_pair_noise(2, lam=2.0)
                for _ in range(400):
                    g.step(1)
                    g.sync()
                out[key] = g.get_state()
                g.close()
        except Exception as e:  # noqa: BLE001
            errors.append(repr(e))

    work("alone")
    assert not errors, errors
    threads = [threading.Thread(target=work, args=(k,)) for k in range(2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
    for k in range(2):
        for x, y in zip(out["alone"], out[k]):
            assert np.array_equal(x, y)
