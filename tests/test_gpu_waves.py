"""Lanes per particle up to the last particle of a wave, and past it, against the
tile kernels of a batch (needs a GPU)."""
import pytest

from test_gpu_lanes import _same, _system

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.set_device(0)


# ends of the waves on 152 SMs: eight, four and two lanes of the one-term form,
# four and two of the general one; four of F^C without and with the VACF
@pytest.mark.parametrize("n,terms,vacf", [
    (14592, "pair", 0), (14593, "pair", 0), (38912, "pair", 40), (38913, "pair", 40), (38913, "pair", 0),
    (14593, "general", 0), (29184, "general", 0), (29185, "general", 40), (58369, "general", 0)])
def test_lanes_give_the_bits_of_the_tile_kernels(n, terms, vacf):
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
