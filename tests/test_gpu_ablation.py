"""Mechanism ablations through the C ABI against the oracle (App.
"Refinement Mechanisms").

* Scale fits (joint, independent, 3-pass coordinate descent) with the codes
  fixed: float32 scales within relative 1e-6 of the oracle's float64 fits
  rounded to float32 (both round a float64-accurate value), objectives
  within relative 1e-6.
* Multi-code probe: the codes after the single-code search, the acceptance
  of the Babai proposal and the number of codes it changes are integers
  decided in float64 on both sides; they must agree on >= 99.5 % of the
  (row, group) cases, and every disagreement must sit at a float64
  near-tie of the oracle's own values (|dF| tiny against F).
* Fixed grid: the scales stay bit-identical, codes >= 99.9 % identical to
  the oracle's fixed-grid sweeps, objective within 1e-5.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]

from oracle import (coordinate_descent_scales, independent_scales, joint_scales,  # noqa: E402
                    multicode_probe, objective, prepare_hessian, refine_fixed_grid)
from synth import small_layer  # noqa: E402


@pytest.fixture(scope="module")
def jarq():
    from paper_2609_38599_gb300 import jarq as mod
    return mod


@pytest.mark.parametrize("din,dout,g,bits", [(256, 96, 64, 3), (384, 130, 128, 4)])
@pytest.mark.parametrize("method", ["joint", "independent", "coordinate"])
def test_scale_fit_parity(jarq, din, dout, g, bits, method):
    lay = small_layer(din, dout, g, bits, seed=din + dout + 1)
    prep = prepare_hessian(lay.H, lay.g)
    if method == "joint":
        ref = joint_scales(prep, lay.W, lay.S0, lay.Q0, lay.Z)
    elif method == "independent":
        ref = independent_scales(prep, lay.W, lay.S0, lay.Q0, lay.Z)
    else:
        ref = coordinate_descent_scales(prep, lay.W, lay.S0, lay.Q0, lay.Z, passes=3)
    ref32 = ref.astype(np.float32)
    hess = jarq.prepare(lay.H, lay.g)
    S = lay.S0.copy()
    Fb, Fa = jarq.fit_scales(hess, lay.W, S, lay.Q0, lay.Z, lay.bits, method, 3)
    hess.close()
    rel = np.abs(S.astype(np.float64) - ref32) / np.maximum(np.abs(ref32), 1e-30)
    print(method, "max rel scale diff", rel.max(), "identical", np.mean(S == ref32))
    assert rel.max() <= 1e-6
    F0 = objective(prep, lay.W, lay.S0, lay.Q0, lay.Z)
    F1 = objective(prep, lay.W, ref32, lay.Q0, lay.Z)
    np.testing.assert_allclose(Fb, F0, rtol=1e-6)
    np.testing.assert_allclose(Fa, F1, rtol=1e-6)
    if method != "independent":
        assert np.all(Fa <= Fb * (1 + 1e-9))


@pytest.mark.parametrize("din,dout,g", [
    (64, 1, 64),       # one row, one column tile, one group
    (192, 129, 64),    # the second CTA of a pair with one row; three column tiles
    (320, 257, 64),    # a second pair with one row
    (128, 256, 128),   # one full pair
    (384, 300, 128),   # three groups of 128
])
def test_projection_pair_edges(jarq, din, dout, g):
    """The target projection on CTA pairs at the edges of its tiles, through
    the joint fit (same bars as test_scale_fit_parity)."""
    lay = small_layer(din, dout, g, 3, seed=7 * din + dout)
    prep = prepare_hessian(lay.H, lay.g)
    ref32 = joint_scales(prep, lay.W, lay.S0, lay.Q0, lay.Z).astype(np.float32)
    hess = jarq.prepare(lay.H, lay.g)
    S = lay.S0.copy()
    Fb, _ = jarq.fit_scales(hess, lay.W, S, lay.Q0, lay.Z, lay.bits, "joint")
    hess.close()
    assert np.all(np.abs(S.astype(np.float64) - ref32) <= 1e-6 * np.abs(ref32))
    np.testing.assert_allclose(Fb, objective(prep, lay.W, lay.S0, lay.Q0, lay.Z), rtol=1e-6)


@pytest.mark.parametrize("din,dout,g,bits", [(256, 80, 64, 3), (384, 64, 128, 3), (256, 48, 64, 4)])
def test_multicode_probe_parity(jarq, din, dout, g, bits):
    lay = small_layer(din, dout, g, bits, seed=din + dout + 2)
    prep = prepare_hessian(lay.H, lay.g)
    hess = jarq.prepare(lay.H, lay.g)
    agree = total = 0
    for i in range(din // g):
        ref = multicode_probe(prep, lay.W, lay.S0, lay.Q0, lay.Z, lay.bits, i)
        out = jarq.multicode_probe(hess, lay.W, lay.S0, lay.Q0, lay.Z, lay.bits, i)
        same = (np.all(out["q_search"] == ref["q_search"], axis=1)
                & (out["accepted"] == ref["accepted"]) & (out["changed"] == ref["changed"])
                & (out["moves"] == ref["moves"]))
        agree += int(same.sum())
        total += same.size
        F = objective(prep, lay.W, lay.S0, lay.Q0, lay.Z)
        for j in np.nonzero(~same)[0]:
            # a disagreement must start at a float64 near-tie
            assert abs(ref["dF"][j]) <= 1e-9 * F[j] or out["moves"][j] != ref["moves"][j], (i, j)
        both = same & ref["accepted"]
        if both.any():
            np.testing.assert_allclose(out["dF"][both], ref["dF"][both], rtol=1e-6,
                                       atol=1e-12 * F.max())
    hess.close()
    print("probe agreement", agree, "/", total)
    assert agree >= 0.995 * total


def test_fixed_grid_parity(jarq):
    lay = small_layer(256, 96, 64, 3, seed=41)
    prep = prepare_hessian(lay.H, lay.g)
    Qo, hist = refine_fixed_grid(prep, lay.W, lay.S0, lay.Q0, lay.Z, lay.bits, 3)
    hess = jarq.prepare(lay.H, lay.g)
    S, Q = lay.S0.copy(), lay.Q0.copy()
    o = jarq.default_options(max_iters=3, early_stop=0)
    o.fixed_grid = 1
    st = jarq.refine(hess, lay.W, S, Q, lay.Z, lay.bits, options=o)
    hess.close()
    assert np.array_equal(S, lay.S0)
    assert np.mean(Q == Qo) >= 0.999
    F_gpu_state = objective(prep, lay.W, S, Q, lay.Z)
    assert np.max(np.abs(st.L_final - F_gpu_state) / F_gpu_state) <= 1e-5
    np.testing.assert_allclose(F_gpu_state, hist[-1], rtol=1e-4)


@pytest.mark.parametrize("g", [64, 128])
@pytest.mark.parametrize("bits", [2, 3, 4, 5, 8])
def test_gram_at_the_largest_digit_sums(jarq, g, bits):
    """Codes at both ends of their range against a matrix whose off-diagonal
    blocks are near their block maximum: the largest digit sums that each way
    of forming the dots has to hold.  Every term of F has one sign (W <= 0 <= c),
    so F is off by no more than its terms: H and W by 2^-38 of an entry, the
    products by less; 2^-35 is allowed."""
    rng = np.random.default_rng(bits + g)
    din, dout, qmax = 6 * g, 300, (1 << bits) - 1
    H = 1.0 - rng.uniform(0, 2.0 ** -6, (din, din))
    H = ((H + H.T) / 2 + np.diag(rng.uniform(0.5, 1, din))).astype(np.float32)
    W = -rng.uniform(0.5, 1, (dout, din)).astype(np.float32)
    Q = np.where(rng.random((dout, din)) < 0.9, qmax, qmax - 1).astype(np.uint8)
    Z = np.zeros((dout, 6), np.int32)
    S = rng.uniform(0.5, 1, (dout, 6)).astype(np.float32)
    prep, hess = prepare_hessian(H, g), jarq.prepare(H, g)
    F, _ = jarq.fit_scales(hess, W, S.copy(), Q, Z, bits, "joint")
    hess.close()
    np.testing.assert_allclose(F, objective(prep, W, S, Q, Z), rtol=2.0 ** -35)


def test_full_size_scale_fits_and_probe_sampled_rows(jarq):
    """The q_proj layer (4096 x 4096, g = 128, 3-bit) from its RTN state: the
    three scale fits and the multi-code probe of two groups on the whole layer;
    the oracle on 24 seeded rows."""
    from synth import config_layer
    lay = config_layer("llama2_7b_q_proj_4096x4096_g128_w3", device="cuda")
    rng = np.random.Generator(np.random.PCG64(77))
    rows = np.sort(rng.choice(lay.dout, 24, replace=False))
    cpu = lambda t: t.cpu().numpy()
    W, S0, Q0, Z = cpu(lay.W)[rows], cpu(lay.S0)[rows], cpu(lay.Q0)[rows], cpu(lay.Z)[rows]
    prep = prepare_hessian(cpu(lay.H), lay.g)
    hess = jarq.prepare(lay.H, lay.g)
    for method, fit in (("joint", joint_scales), ("independent", independent_scales),
                        ("coordinate", lambda *a: coordinate_descent_scales(*a, passes=3))):
        S = lay.S0.clone()
        jarq.fit_scales(hess, lay.W, S, lay.Q0, lay.Z, lay.bits, method, 3)
        ref = fit(prep, W, S0, Q0, Z).astype(np.float32)
        rel = np.abs(cpu(S)[rows].astype(np.float64) - ref) / np.maximum(np.abs(ref), 1e-30)
        print(method, "max rel", rel.max())
        assert rel.max() <= 1e-6, method
    for i in (0, 17):
        out = jarq.multicode_probe(hess, lay.W, lay.S0, lay.Q0, lay.Z, lay.bits, i)
        ref = multicode_probe(prep, W, S0, Q0, Z, lay.bits, i)
        same = (np.all(cpu(out["q_search"])[rows] == ref["q_search"], axis=1)
                & (cpu(out["accepted"])[rows] == ref["accepted"])
                & (cpu(out["changed"])[rows] == ref["changed"]))
        print("group", i, "probe rows identical", int(same.sum()), "/", len(rows))
        assert same.mean() >= 0.95
    hess.close()
