"""The FP64 / FP32 embedding as digit products (emb_digits.cu) against the FP64 oracle at the edges of its
16-row tiles, over the weight ranges of its fixed-point layers and beyond them (GPU only).

Bars, from the arithmetic: FP64 keeps 54 bits of every operand, so per-atom energies agree to the 1e-10 of the
other FP64 tests and forces to 1e-9 of their rms; weights 40 times larger carry 40 times the absolute error of
the sums into tanh and its slope (1e-8, 1e-6), weights beyond the fixed-point range take the plain kernels.
FP32: about 100 terms a sum at 6e-8 each, 6e-6, with a factor of ten for the forces' cancellation."""
import numpy as np
import pytest

import oracle
from paper_2410_22867_gb300 import synth

from _parity import errors

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _cluster(n, seed):
    """n atoms of two types within 4.8 A of each other (all pairs inside r_c 6 A) in a 30 A box."""
    rng = np.random.default_rng(seed)
    x = []
    while len(x) < n:
        p = rng.uniform(-2.4, 2.4, 3)
        if np.linalg.norm(p) < 2.4 and all(np.linalg.norm(p - q) > 0.55 for q in x):
            x.append(p)
    types = (np.arange(n) % 3 > 0).astype(np.int32)
    return np.array(x).reshape(n, 3) + 15.0, types, np.diag([30.0] * 3).reshape(-1)


def _weights(scale):
    w = synth.xavier_weights(("O", "H"), 6.0, 0.5, (46, 92), 1001)
    for ti in range(2):
        for tj in range(2):
            for name in ("W2", "W3"):
                w.block(f"emb{ti}{tj}.{name}")[...] *= scale
    return w


@pytest.mark.parametrize("prec,scale,e_bar,f_bar", [("fp64", 1.0, 1e-10, 1e-9), ("fp64", 40.0, 1e-8, 1e-6),
                                                    ("fp64", 1e6, 1e-8, None), ("fp32", 1.0, 6e-6, 6e-5)])
@pytest.mark.parametrize("n", [1, 2, 16, 17, 25, 26, 49, 50, 66])
def test_tiles_and_weight_ranges(prec, scale, e_bar, f_bar, n):
    import paper_2410_22867_gb300 as dp
    x, t, box = _cluster(n, n)
    w = _weights(scale)
    ref = oracle.Model(w.to_blob()).compute(x, t, box)
    m = dp.DPModel(w, prec, max_atoms=n)
    out = m.compute(torch.tensor(x, device="cuda"), torch.tensor(t, device="cuda"), box)
    e = errors(out, ref, t)
    assert e["ei_rel"] <= e_bar, e
    if n == 1:
        assert float(out["forces"].abs().max()) == 0.0
    elif f_bar is not None:
        assert e["f_rel"] <= f_bar, e
