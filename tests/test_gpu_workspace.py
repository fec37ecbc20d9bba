"""A mechanism's device workspace is what its kernels can reach."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not torch.cuda.is_available(),
                                                  reason="needs a CUDA GPU")]

from paper_1607_03884_gb300 import kin, synth  # noqa: E402


@pytest.mark.parametrize("form", [kin.Mechanism, kin.ConcMechanism])
def test_slots_of_a_large_mechanism(form):
    """53 species: four teams per SM, each with a Jacobian and a complex matrix
    of at most 54 unknowns in FP64; tables and counters below 1 MB."""
    ch4, sms = synth.make_mechanism("ch4"), torch.cuda.get_device_properties(0).multi_processor_count
    first = form(ch4)  # what the first handle of a process sets up besides
    before = torch.cuda.mem_get_info()[0]
    second = form(ch4)
    used = before - torch.cuda.mem_get_info()[0]
    # allocations round up to 2 MiB pages
    assert used <= sms * 4 * 3 * 54 * 55 * 8 + (1 << 20) + 8 * (2 << 20), used
    del first, second
