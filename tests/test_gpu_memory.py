"""Device memory that a model takes (GPU only): the parameter gradient's fitting activations and neighbour rows share
one area, since they are never in use together.  2,048 water atoms in FP32, from the allocations of dp_create: about
33 KB an atom of lists and evaluation buffers (65 MiB), the weights and their copies (30 MiB), the gradient's two
T arrays (12.5 MiB) and the larger of its areas, 32,768 rows of 709 values (89 MiB): 197 MiB, and 10% for the
granularity of the allocations."""
import pytest

from paper_2410_22867_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_gradient_areas_are_shared():
    import paper_2410_22867_gb300 as dp
    dp.DPModel(synth.water_weights(), "fp32", max_atoms=64).close()  # what is allocated once per process
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    m = dp.DPModel(synth.water_weights(), "fp32", max_atoms=2048)
    taken = before - torch.cuda.mem_get_info()[0]
    m.close()
    assert taken <= 217 * 2 ** 20, taken / 2 ** 20
