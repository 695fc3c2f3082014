"""New parameters for a tabulated model whose MD steps are captured: the table is rebuilt where it is, so that the
captured steps read the new one (GPU only).  Bars: the order of atomic force sums over 4 steps, as in
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
