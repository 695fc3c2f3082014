"""dp_set_params_device (parameters that live on the GPU) against dp_set_params, and its refusals (GPU only).
The same parameters give the same device copies, so results agree to the run-to-run order of atomic sums
(1e-12 in FP64, 1e-5 in FP32, 1e-3 in mixed precision, of the forces' norm)."""
import numpy as np
import pytest

from paper_2410_22867_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,bar", [("fp64", 1e-12), ("fp32", 1e-5), ("mix_fp16", 1e-3)])
@pytest.mark.parametrize("dtype", ["float32", "float64"])
@pytest.mark.parametrize("own_stream", [False, True])
def test_device_parameters(prec, bar, dtype, own_stream):
    import paper_2410_22867_gb300 as dp
    s = synth.water_box(64, 4)
    a, b = synth.water_weights(1001), synth.water_weights(7)
    th = torch.tensor(b.theta, dtype=getattr(torch, dtype))
    stream = torch.cuda.Stream() if own_stream else None
    x = torch.tensor(s.coords, device="cuda")
    t = torch.tensor(s.types, device="cuda")
    torch.cuda.synchronize()
    m1 = dp.DPModel(a, prec, max_atoms=s.natoms, stream=stream)
    m2 = dp.DPModel(a, prec, max_atoms=s.natoms, stream=stream)
    m1.set_params(th)                  # host path
    m2.set_params(th.to("cuda"))       # device path
    o1, o2 = m1.compute(x, t, s.box), m2.compute(x, t, s.box)
    d = float((o1["forces"] - o2["forces"]).norm() / o1["forces"].norm())
    assert d <= bar
    assert abs(float(o1["energy"]) - float(o2["energy"])) <= bar * abs(float(o1["energy"]))
    # a strided view goes through the host as before
    wide = torch.stack([th, th], 1).to("cuda")
    m2.set_params(wide[:, 0])
    o3 = m2.compute(x, t, s.box)
    assert float((o1["forces"] - o3["forces"]).norm() / o1["forces"].norm()) <= bar
    bad = th.to("cuda").clone()
    bad[12345] = float("nan")
    with pytest.raises(dp.DPError) as e:
        m2.set_params(bad)
    assert e.value.status == 9
    with pytest.raises(dp.DPError) as e:
        m2.set_params(th.to("cuda")[:-1])
    assert e.value.status == 1
    o4 = m2.compute(x, t, s.box)       # the refused parameters left the model as it was
    assert float((o1["forces"] - o4["forces"]).norm() / o1["forces"].norm()) <= bar
