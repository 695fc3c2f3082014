"""The shared-memory table kernels of the mixed precisions (tab_mix.cu) against the oracle's tables, at the
table sizes around what shared memory holds (318 intervals; 319 take the other kernels), in a box, a sheared
box and a batch whose replicas end inside a warp's atoms (GPU only).

Bars: the mixed precisions' relative errors on the normalised water model (the other kernels' bars)."""
import numpy as np
import pytest

import oracle
from paper_2410_22867_gb300 import synth

from _parity import env_stats, errors
from test_gpu_normalised import BARS

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SHEAR = np.array([[1.0, 0.0, 0.0], [0.1, 1.0, 0.0], [-0.05, 0.07, 1.0]])


@pytest.mark.parametrize("n", [2, 256, 318, 319])
@pytest.mark.parametrize("prec", ["mix_bf16", "mix_fp16"])
@pytest.mark.parametrize("form", ["box", "sheared", "batch"])
def test_table_forms(prec, n, form):
    import paper_2410_22867_gb300 as dp
    w = synth.normalised_weights("water", env_stats())
    systems = [synth.water_box(m, 5 + m) for m in ((33, 140, 77) if form == "batch" else (250,))]
    if form == "sheared":
        for s in systems:
            s.coords = s.coords @ SHEAR
            s.box = (s.box.reshape(3, 3) @ SHEAR).reshape(-1)
    coords, types, offs, boxes = synth.concat(systems)
    assert len(types) * sum(w.sel) >= 100000  # the shared-memory kernels' range
    m = dp.DPModel(w, prec, max_atoms=len(types), max_replicas=len(systems))
    x0, x1, _ = m.tabulate(n)
    orc = oracle.Model(w.to_blob())
    orc.tabulate(x0, x1, n)
    out = m.compute_batch(torch.tensor(coords, device="cuda"), torch.tensor(types, device="cuda"), offs, boxes)
    for k, s in enumerate(systems):
        ref = orc.compute(s.coords, s.types, s.box)
        of = slice(int(offs[k]), int(offs[k + 1]))
        e = errors({q: out[q][of] for q in ("forces", "atom_energy")}, ref, s.types)
        bar = BARS["water"][prec]
        if n > 2:  # two intervals are no approximation of the net: large slopes, absolute comparison only
            assert e["f_rel"] <= bar["f_rel"], e
            assert e["dev_rel"] <= bar["dev_rel"], e
            v = out["virial"][k].cpu().numpy()
            assert np.abs(v - ref["virial"]).max() <= 2e-2 * np.abs(ref["virial"]).max()
        else:
            assert e["f_rel"] <= 5 * bar["f_rel"], e
    m.close()


@pytest.mark.parametrize("prec", ["mix_bf16", "mix_fp16"])
def test_rows_outside_the_table(prec):
    """A table that ends below the bonded O-H pairs: their rows (about 700) lie up to 98 intervals beyond
    the last node and take the edge interval's polynomial, which is within 0.015 of the net there (outputs of
    up to 2.9), so the same bars hold."""
    import paper_2410_22867_gb300 as dp
    w = synth.normalised_weights("water", env_stats())
    s = synth.water_box(250, 255)
    m = dp.DPModel(w, prec, max_atoms=s.natoms)
    x0, x1, _ = m.tabulate(256)
    x1 = x0 + 0.48 * (x1 - x0)
    m.tabulate(256, x0, x1)
    orc = oracle.Model(w.to_blob())
    orc.tabulate(x0, x1, 256)
    out = m.compute(torch.tensor(s.coords, device="cuda"), torch.tensor(s.types, device="cuda"), s.box)
    ref = orc.compute(s.coords, s.types, s.box)
    e = errors({q: out[q] for q in ("forces", "atom_energy")}, ref, s.types)
    bar = BARS["water"][prec]
    assert e["f_rel"] <= bar["f_rel"], e
    assert e["dev_rel"] <= bar["dev_rel"], e
    m.close()
