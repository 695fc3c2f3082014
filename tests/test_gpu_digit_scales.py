"""FP64 / FP32 nets whose weights or activations spread widely, against the FP64 oracle (GPU only).

The digit products hold every operand relative to a scale, so what a scale covers (a column of weights, a row of
activations) decides how many bits the small values keep.  Bars as for evenly scaled nets, from the arithmetic.
FP32: about 100 terms a sum at 6e-8 each, 6e-6 on energies, with a factor of ten for the forces' cancellation.
FP64: 1.1e-16 a rounding, sums of up to 1,600 terms (a random walk of 40) on both sides: 2e-14 on energies,
a factor of ten for the forces."""
import numpy as np
import pytest

import oracle
from paper_2410_22867_gb300 import synth

from _parity import errors
from test_gpu_digits import _cluster

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

BARS = {"fp64": (2e-14, 2e-13), "fp32": (6e-6, 6e-5)}


def _pairs():
    return [(ti, tj) for ti in range(2) for tj in range(2)]


def _check(w, prec, n=66, seed=66):
    import paper_2410_22867_gb300 as dp
    x, t, box = _cluster(n, seed)
    ref = oracle.Model(w.to_blob()).compute(x, t, box)
    m = dp.DPModel(w, prec, max_atoms=n)
    e = errors(m.compute(torch.tensor(x, device="cuda"), torch.tensor(t, device="cuda"), box), ref, t)
    m.close()
    assert e["ei_rel"] <= BARS[prec][0] and e["f_rel"] <= BARS[prec][1], e


def _outlier(layer, value):
    """One weight of W2 or W3 of every pair far above the others.  Its input (unit 3) is a constant, so that its
    output is saturated and the other columns decide the result; columns 9 are far below the others."""
    w = synth.xavier_weights(("O", "H"), 6.0, 0.5, (46, 92), 1001)
    for ti, tj in _pairs():
        b = {k: w.block(f"emb{ti}{tj}.{k}") for k in ("W1", "b1", "W2", "b2", "W3", "b3")}
        b["W1"][0, 3], b["b1"][3] = 0.0, 1.0
        b["W2"][:, 3], b["b2"][3] = 0.0, 1.0
        b["W2"][:, 9] *= 1e-6
        b["W3"][:, 9] *= 1e-6
        b[layer][3, 7] = value
    return w


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("layer", ["W2", "W3"])
@pytest.mark.parametrize("value", [100.0, 16384.0])
def test_one_large_embedding_weight_of_a_live_unit(prec, layer, value):
    """As above, but unit 3 varies (its activations stay above 0.6): its gradient is a sum in which the large weight
    meets the zero gradient of the output that it saturates."""
    w = _outlier(layer, value)
    for ti, tj in _pairs():
        b = {k: w.block(f"emb{ti}{tj}.{k}") for k in ("W1", "b1", "W2", "b2")}
        b["W1"][0, 3], b["b1"][3] = -0.4, 1.5
        b["W2"][:, 3], b["b2"][3] = b["W2"][:, 4] * 0.3, 2.0
    _check(w, prec)


# 0.3: the digit products; from 100 on the plain kernels (the spread of the column, beyond 65,536 the size too)
@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("layer", ["W2", "W3"])
@pytest.mark.parametrize("value", [0.3, 100.0, 16384.0, 65535.0, 65600.0])
def test_one_large_embedding_weight(prec, layer, value):
    _check(_outlier(layer, value), prec)


def _small(w1, fit):
    """Activations of about w1 times the input in every row: no embedding biases, small first-layer weights; the fitting
    nets' first layer scaled to match."""
    w = synth.xavier_weights(("O", "H"), 6.0, 0.5, (46, 92), 1001)
    for ti, tj in _pairs():
        w.block(f"emb{ti}{tj}.W1")[...] *= w1
        for k in ("b1", "b2", "b3"):
            w.block(f"emb{ti}{tj}.{k}")[...] = 0.0
    for t in range(2):
        w.block(f"fit{t}.W1")[...] *= fit
    return w


@pytest.mark.parametrize("w1,fit", [(0.1, 1e3), (1e-2, 1e5), (1e-4, 1e9)])
def test_small_activations_fp32(w1, fit):
    _check(_small(w1, fit), "fp32")


# 3 (rms of h1 0.25): the fixed-point layers; the others: the plain kernels
@pytest.mark.parametrize("w1,fit", [(3.0, 10.0), (0.1, 1e3), (1e-2, 1e5), (1e-4, 1e9)])
def test_small_activations_fp64(w1, fit):
    _check(_small(w1, fit), "fp64")


def _fit_outlier(layer, value):
    """One large weight in W1, W2 or W3 of both fitting nets whose input is never near zero (D_00 = |T_0|^2; units 3
    made constant), so that its output is saturated; columns 9 far below the others."""
    w = synth.xavier_weights(("O", "H"), 6.0, 0.5, (46, 92), 1001, fit_gain=10.0)
    for t in range(2):
        b = {k: w.block(f"fit{t}.{k}") for k in ("W1", "b1", "W2", "b2", "W3")}
        b["W1"][:, 3], b["b1"][3] = 0.0, 1.0
        b["W2"][:, 3], b["b2"][3] = 0.0, 1.0
        for k in ("W1", "W2", "W3"):
            b[k][:, 9] *= 1e-6
        b[layer][0 if layer == "W1" else 3, 7] = value
    return w


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("layer", ["W1", "W2", "W3"])
@pytest.mark.parametrize("value", [1e5, 1e8])
@pytest.mark.parametrize("n", [66, 3])
def test_one_large_fitting_weight(prec, layer, value, n):
    _check(_fit_outlier(layer, value), prec, n, n)


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
def test_one_large_descriptor_element(prec):
    """D_00 about 1, the rest of its rows 1e-2 and 1e-4: embedding output 0 is near 1, the others near 1e-2."""
    w = _small(1e-2, 100.0)
    for ti, tj in _pairs():
        w.block(f"emb{ti}{tj}.b3")[0] = 5.0
    _check(w, prec)


def test_infinite_fp32_weight():
    """A parameter beyond FP32 makes a column infinite: its unit is saturated as in the oracle's FP64."""
    import paper_2410_22867_gb300 as dp
    x, t, box = _cluster(16, 16)
    w = synth.xavier_weights(("O", "H"), 6.0, 0.5, (46, 92), 1001)
    w.block("fit0.W2")[5, 5] = 1e300
    ref = oracle.Model(w.to_blob()).compute(x, t, box)["atom_energy"]
    m = dp.DPModel(w, "fp32", max_atoms=16)
    e = m.compute(torch.tensor(x, device="cuda"), torch.tensor(t, device="cuda"), box)["atom_energy"].cpu().numpy()
    assert np.abs(e - ref).max() <= BARS["fp32"][0] * np.abs(ref).mean()


def test_captured_steps_follow_the_kernels():
    """MD steps captured with one set of kernels are captured again when new parameters need the other one."""
    import paper_2410_22867_gb300 as dp
    s = synth.water_box(64, 3)
    inside = synth.water_weights(1001)
    outside = synth.water_weights(1001)
    for ti, tj in _pairs():
        b = {k: outside.block(f"emb{ti}{tj}.{k}") for k in ("W1", "b1", "W2")}
        b["W1"][0, 3], b["b1"][3] = 0.0, 1.0
        b["W2"][3, 7] = 1e5
    v0 = synth.maxwell_boltzmann(s.masses()[s.types], 300.0, 5)
    types = torch.tensor(s.types, device="cuda")

    def run(m):
        x, v = torch.tensor(s.coords, device="cuda"), torch.tensor(v0, device="cuda")
        k = m.verlet(m.md_state(x, v, types, s.box, s.masses(), rebuild_every=2), 0.5, 4)
        return k["forces"].clone(), k["potential"].clone()

    m = dp.DPModel(inside, "fp64", max_atoms=s.natoms)
    wide = synth.water_weights(1001)
    for k in range(2):
        wide.block(f"fit{k}.W2")[3, 7] = 100.0
    for w in (inside, outside, wide, inside):
        m.set_params(w.theta)
        f, e = run(m)
        fresh = dp.DPModel(w, "fp64", max_atoms=s.natoms)
        f1, e1 = run(fresh)
        assert float((f - f1).norm() / f1.norm()) <= 1e-11  # order of the atomic sums, 4 steps
        assert abs(float(e - e1)) <= 1e-12 * abs(float(e1))
        fresh.close()


def _small_fit(gain):
    """Fitting activations of about `gain`: no fitting biases, first-layer weights scaled down."""
    w = synth.xavier_weights(("O", "H"), 6.0, 0.5, (46, 92), 1001)
    for t in range(2):
        w.block(f"fit{t}.W1")[...] *= gain
        for k in ("b1", "b2", "b3", "b4"):
            w.block(f"fit{t}.{k}")[...] = 0.0
    return w


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("gain", [1e-2, 1e-4, 1e-6])
def test_small_fitting_activations(prec, gain):
    _check(_small_fit(gain), prec)


@pytest.mark.parametrize("n", [64, 256])
def test_fp32_force_sums_are_fp64(n):
    """The net force of an FP32 model: every pair force enters with both signs, and sums in FP64 of 24-bit values (29 bits
    to spare) are exact but for the pairs 2^-29 below the largest.  Bar: a fiftieth of what one rounding of the
    largest force at every addition (two a neighbour, about 95 neighbours) would leave as a random walk."""
    import paper_2410_22867_gb300 as dp
    from _parity import env_stats
    s = synth.water_box(n, 1)
    m = dp.DPModel(synth.normalised_weights("water", env_stats()), "fp32", max_atoms=s.natoms)
    f = m.compute(torch.tensor(s.coords, device="cuda"), torch.tensor(s.types, device="cuda"), s.box)["forces"].cpu().numpy()
    net = np.abs(f.astype(np.longdouble).sum(0)).max()
    assert float(net) <= 0.02 * 2.0 ** -53 * np.sqrt(2 * 95 * s.natoms) * np.abs(f).max()


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("nmol", [21, 22, 64, 65])
def test_plain_kernels_in_a_box(prec, nmol):
    """Both nets by FMAs, at the edges of the fitting GEMM's 64-row blocks (one, two and three of hydrogens)."""
    import paper_2410_22867_gb300 as dp
    s = synth.water_box(nmol, nmol)
    w = synth.xavier_weights(("O", "H"), 6.0, 0.5, (46, 92), 1001, fit_gain=10.0)
    for ti, tj in _pairs():
        w.block(f"emb{ti}{tj}.W3")[3, 7] = 3.0
    for t in range(2):
        w.block(f"fit{t}.W2")[3, 7] = 2.0
    ref = oracle.Model(w.to_blob()).compute(s.coords, s.types, s.box)
    m = dp.DPModel(w, prec, max_atoms=s.natoms)
    e = errors(m.compute(torch.tensor(s.coords, device="cuda"), torch.tensor(s.types, device="cuda"), s.box), ref, s.types)
    m.close()
    assert e["ei_rel"] <= BARS[prec][0] and e["f_rel"] <= BARS[prec][1], e


# 40 times larger embedding weights carry 40 times the error of the sums; at 1e6 (plain kernels) tanh is a step whose rare
# unsaturated places carry 1e6 times it
@pytest.mark.parametrize("prec,scale,f_bar", [("fp32", 40.0, 40 * BARS["fp32"][1]), ("fp64", 1e6, 1e6 * BARS["fp64"][1])])
def test_forces_of_large_embedding_weights(prec, scale, f_bar):
    import paper_2410_22867_gb300 as dp
    from test_gpu_digits import _weights
    x, t, box = _cluster(66, 66)
    w = _weights(scale)
    ref = oracle.Model(w.to_blob()).compute(x, t, box)
    m = dp.DPModel(w, prec, max_atoms=66)
    e = errors(m.compute(torch.tensor(x, device="cuda"), torch.tensor(t, device="cuda"), box), ref, t)
    m.close()
    assert e["ei_rel"] <= 40 * BARS["fp32"][0] and e["f_rel"] <= f_bar, e


@pytest.mark.parametrize("kind", ["even", "outlier", "small"])
@pytest.mark.parametrize("nt", [3, 4])
def test_many_types_fp64(kind, nt):
    """FP64 models of three atom types are the largest that the plain embedding kernels hold; with four, digits take them
    whatever their spread (bars of the other FP64 tests)."""
    import paper_2410_22867_gb300 as dp
    x, t, box = _cluster(40, 40)
    t = (np.arange(40) % nt).astype(np.int32)
    w = synth.xavier_weights(tuple("ABCD"[:nt]), 6.0, 0.5, (20,) * nt, 1001)
    for ti in range(nt):
        for tj in range(nt):
            if kind == "outlier":
                w.block(f"emb{ti}{tj}.W3")[3, 7] = 100.0
            if kind == "small":
                w.block(f"emb{ti}{tj}.W1")[...] *= 1e-2
                for k in ("b1", "b2", "b3"):
                    w.block(f"emb{ti}{tj}.{k}")[...] = 0.0
    ref = oracle.Model(w.to_blob()).compute(x, t, box)
    m = dp.DPModel(w, "fp64", max_atoms=40)
    e = errors(m.compute(torch.tensor(x, device="cuda"), torch.tensor(t, device="cuda"), box), ref, t)
    m.close()
    assert e["ei_rel"] <= 1e-10 and e["f_rel"] <= 1e-9, e


def test_a_refused_launch_leaves_other_models_alone():
    """FP64 tables of four types do not fit shared memory: that model's call is refused, another model's calls run."""
    import paper_2410_22867_gb300 as dp
    x, t, box = _cluster(16, 16)
    x, box0 = torch.tensor(x, device="cuda"), box
    four = dp.DPModel(synth.xavier_weights(tuple("ABCD"), 6.0, 0.5, (20,) * 4, 1001), "fp64", max_atoms=16)
    four.tabulate(16)
    other = dp.DPModel(synth.xavier_weights(("O", "H"), 6.0, 0.5, (46, 92), 1001), "fp64", max_atoms=16)
    tt = torch.tensor(t, device="cuda")
    with pytest.raises(dp.DPError):
        four.compute(x, tt, box0)
    e = other.compute(x, tt, box0)["energy"]
    assert torch.isfinite(e).all()
    dp.DPModel(synth.water_weights(), "fp32", max_atoms=16).close()
