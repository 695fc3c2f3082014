"""Device memory that a model takes (GPU only): the parameter gradient's fitting activations and neighbour rows share
one area, since they are never in use together.  2,048 water atoms in FP32, from the allocations of dp_create: about
33 KB an atom of lists and evaluation buffers (65 MiB), the weights and their copies (30 MiB), the gradient's two
T arrays (12.5 MiB) and the larger of its areas, 32,768 rows of 709 values (89 MiB): 197 MiB, and 10% for the
granularity of the allocations."""
import gc

import pytest

from paper_2410_22867_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_gradient_areas_are_shared():
    import paper_2410_22867_gb300 as dp
    gc.collect()  # models of other tests
    dp.DPModel(synth.water_weights(), "fp32", max_atoms=64).close()  # what is allocated once per process
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    m = dp.DPModel(synth.water_weights(), "fp32", max_atoms=2048)
    taken = before - torch.cuda.mem_get_info()[0]
    m.close()
    assert taken <= 217 * 2 ** 20, taken / 2 ** 20


def test_reduction_slots_of_many_replicas():
    """4,096 replicas of up to 131,072 atoms: the partial sums take 4,096 x 17 slots of 80 B (5.3 MiB), the replicas'
    geometry, cells and results 6 MiB more than one replica's; 14 MiB with the granularity of the allocations.  One
    box of 5,000 molecules among them, and sums over it and its neighbours."""
    import numpy as np

    import paper_2410_22867_gb300 as dp
    w = synth.xavier_weights(("O", "H"), 3.0, 0.5, (8, 16), 1001)

    def taken(reps):
        gc.collect()
        torch.cuda.synchronize()
        before = torch.cuda.mem_get_info()[0]
        m = dp.DPModel(w, "fp32", max_atoms=131072, max_replicas=reps, skin=0.5)
        return m, before - torch.cuda.mem_get_info()[0]

    m, one = taken(1)
    m.close()
    m, many = taken(4096)
    assert many - one <= 14 * 2 ** 20, (many - one) / 2 ** 20
    # 600 replicas, one of them 15,000 atoms: chunks larger than a single box's
    systems = [synth.water_box(5000 if k == 300 else 8, k) for k in range(600)]
    coords, types, offs, boxes = synth.concat(systems)
    m.set_truncation(True)
    out = m.compute_batch(torch.tensor(coords, device="cuda"), torch.tensor(types, device="cuda"), offs, boxes)
    ea = out["atom_energy"].cpu().numpy()
    e = out["energy"].cpu().numpy()
    want = np.array([ea[a:b].sum() for a, b in zip(offs[:-1], offs[1:])])
    assert np.abs(e - want).max() <= 1e-12 * np.abs(want).max()  # FP64 sums of the same values
    f = out["forces"].cpu().numpy()
    assert np.isfinite(f).all() and np.isfinite(out["virial"].cpu().numpy()).all()
    m.close()
