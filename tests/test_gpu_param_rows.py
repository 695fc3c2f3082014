"""The parameter gradient's row-chunked layers against the oracle's dual-number gradient at the edges of their
tiles: centres without neighbours of a type, row counts around the 128- and 256-row blocks (GPU only).

Bars: FP64 gradients are sums of at most 10^4 terms of FP64 products, 1e-10 of the gradient's norm as in the
other parameter-gradient tests; FP32 the same sums at 6e-8 a term, random in sign, 1e-4 of the norm."""
import numpy as np
import pytest

import oracle
from paper_2410_22867_gb300 import synth

from _parity import env_stats

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,bar", [("fp64", 1e-10), ("fp32", 1e-4)])
@pytest.mark.parametrize("n_o,n_h", [(1, 0), (2, 0), (1, 2), (12, 11), (16, 17), (5, 40)])
def test_gradient_rows(prec, bar, n_o, n_h):
    import paper_2410_22867_gb300 as dp
    n = n_o + n_h
    rng = np.random.default_rng(100 * n_o + n_h)
    x = []
    while len(x) < n:  # a cluster: every atom sees every other
        p = rng.uniform(-2.4, 2.4, 3)
        if np.linalg.norm(p) < 2.4 and all(np.linalg.norm(p - q) > 0.6 for q in x):
            x.append(p)
    x = np.array(x).reshape(n, 3) + 15.0
    t = np.array([0] * n_o + [1] * n_h, dtype=np.int32)
    box = np.diag([30.0] * 3).reshape(-1)
    w = synth.normalised_weights("water", env_stats())
    F0 = rng.normal(0.0, 0.5, size=(n, 3))
    # 12 parameters of every embedding net (each layer's weights and biases) and 6 of each fitting net
    idx = []
    for name, shape, off in synth.theta_layout(2)[0]:
        size = int(np.prod(shape))
        idx += [off + int(q) for q in rng.choice(size, size=min(size, 2 if name.startswith("emb") else 1), replace=False)]
    idx = np.array(sorted(idx))
    ref, _, ref_loss = oracle.Model(w.to_blob()).param_grad(x, t, box, 0.3, F0, idx, 0.7, 0.2)
    m = dp.DPModel(w, prec, max_atoms=n)
    g, loss = m.param_grad(torch.tensor(x, device="cuda"), torch.tensor(t, device="cuda"), box, 0.3,
                           torch.tensor(F0, device="cuda"), 0.7, 0.2)
    d = g.cpu().numpy()[idx] - ref
    assert np.linalg.norm(d) <= bar * np.linalg.norm(ref)
    assert abs(float(loss) - ref_loss) <= bar * abs(ref_loss)
