"""Tabulated models: new parameters while MD steps are captured (the table is rebuilt where it is, so that the captured
steps read the new one), and the autotuner (GPU only).  Bars: the order of atomic force sums over 4 steps, as in
test_gpu_params_device.py."""
import pytest

from paper_2410_22867_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,bar", [("fp64", 1e-11), ("mix_fp16", 1e-3)])
def test_captured_steps_use_the_new_table(prec, bar):
    import paper_2410_22867_gb300 as dp
    s = synth.water_box(64, 3)
    types = torch.tensor(s.types, device="cuda")
    v0 = synth.maxwell_boltzmann(s.masses()[s.types], 300.0, 5)

    def run(m):
        x, v = torch.tensor(s.coords, device="cuda"), torch.tensor(v0, device="cuda")
        k = m.verlet(m.md_state(x, v, types, s.box, s.masses(), rebuild_every=2), 0.5, 4)
        return k["forces"].clone()

    a, b = synth.water_weights(1001), synth.water_weights(7)
    m = dp.DPModel(a, prec, max_atoms=s.natoms)
    m.tabulate(256)
    run(m)  # captures the steps
    held = []
    for w in (b, a, b):
        held.append(torch.empty(1 << 20, device="cuda"))  # other memory moves between the rebuilds
        m.set_params(w.theta)
        f = run(m)
        fresh = dp.DPModel(w, prec, max_atoms=s.natoms)
        fresh.tabulate(256)
        f1 = run(fresh)
        assert float((f - f1).norm() / f1.norm()) <= bar
        fresh.close()
    m.tabulate(64)  # another size: a new table, steps captured again
    f = run(m)
    fresh = dp.DPModel(b, prec, max_atoms=s.natoms)
    fresh.tabulate(64)
    f1 = run(fresh)
    assert float((f - f1).norm() / f1.norm()) <= bar


def test_autotune_leaves_kernels_of_one_shape():
    """The shared-memory table kernels have one launch shape: nothing is tuned for them; below their range it is."""
    import paper_2410_22867_gb300 as dp
    for cells, large in ((6, True), (3, False)):
        s = synth.copper_fcc(cells, 1)
        m = dp.DPModel(synth.copper_weights(1001), "mix_fp16", max_atoms=s.natoms)
        m.tabulate(256)
        x, t = torch.tensor(s.coords, device="cuda"), torch.tensor(s.types, device="cuda")
        f0 = m.compute(x, t, s.box)["forces"]
        g = m.autotune(1)
        assert g[2] > 0 and g[3] > 0 and (g[0] > 0) != large and (g[1] > 0) != large, g
        f1 = m.compute(x, t, s.box)["forces"]
        assert float((f0 - f1).norm() / f0.norm()) <= 1e-3  # as test_gpu_params_device.py's mixed bar
        m.close()
