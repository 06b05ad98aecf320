"""Write-back post-passes and the ridge-acceptance variant on the GPU,
against the oracle (bit-exact for the integer and rounding work).

App. E "Representing Negative Scales" (Eq. canonicalization), App. E "Early
stopping" (the refined weights cast to the model's dtype), Sec. 3.1 (b-bit
codes), App. G Remark ridge-acceptance.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]

from oracle import (Options, canonicalize, dequantize_cast, pack_codes, prepare_hessian,  # noqa: E402
                    refine_layer, scale_system)
from synth import small_layer  # noqa: E402


@pytest.fixture(scope="module")
def jarq():
    from paper_2609_38599_gb300 import jarq as J
    return J


def _signed_state(dout, din, g, bits, seed):
    rng = np.random.default_rng(seed)
    G = din // g
    S = (rng.standard_normal((dout, G)) * 0.01).astype(np.float32)   # about half negative
    Q = rng.integers(0, 1 << bits, size=(dout, din), dtype=np.uint8)
    Z = rng.integers(0, 1 << bits, size=(dout, G)).astype(np.int32)
    return S, Q, Z


@pytest.mark.parametrize("dout,din,g,bits", [(130, 384, 128, 3), (77, 192, 64, 4), (5, 96, 32, 8)])
def test_canonicalize_bit_exact(jarq, dout, din, g, bits):
    S, Q, Z = _signed_state(dout, din, g, bits, seed=dout)
    S2, Q2, Z2 = canonicalize(S.astype(np.float64), Q, Z, bits)
    t = lambda a: torch.as_tensor(a).cuda()
    Sd, Qd, Zd = t(S), t(Q), t(Z)
    jarq.canonicalize(Sd, Qd, Zd, g, bits)
    assert np.array_equal(Sd.cpu().numpy(), S2.astype(np.float32))
    assert np.array_equal(Qd.cpu().numpy(), Q2)
    assert np.array_equal(Zd.cpu().numpy(), Z2)
    assert (S2 >= 0).all()


@pytest.mark.parametrize("dtype", ["float32", "float16", "bfloat16"])
def test_dequantize_bit_exact(jarq, dtype):
    S, Q, Z = _signed_state(96, 256, 64, 4, seed=9)
    ref = dequantize_cast(S, Q, Z, 64, dtype)
    t = lambda a: torch.as_tensor(a).cuda()
    out = jarq.dequantize(t(S), t(Q), t(Z), 64, 4, dtype).float().cpu().numpy().astype(np.float64)
    assert np.array_equal(out, np.asarray(ref, dtype=np.float64))


def _offset_copy(a, off):
    """A contiguous device copy of `a` whose data starts `off` elements into its storage."""
    t = torch.as_tensor(a)
    buf = torch.empty(t.numel() + off, dtype=t.dtype, device="cuda")[off:].view(t.shape)
    return buf.copy_(t)


@pytest.mark.parametrize("dtype", ["float32", "float16", "bfloat16"])
@pytest.mark.parametrize("g,off", [(64, 0), (64, 1), (48, 0), (24, 0)])
def test_dequantize_rounds_once_over_the_whole_range(jarq, dtype, g, off):
    """The 16-code and the single-code kernel (misaligned codes, g not a
    multiple of 16) on scales from subnormal to overflowing, products at and
    next to ties: one rounding of the exact product."""
    rng = np.random.default_rng(g + off)
    dout, din, bits = 67, 8 * g, 8
    G = din // g
    e = rng.integers(-40, 20, size=(dout, G)).astype(np.float64)
    # the oracle's bfloat16 rounding has no subnormals and no overflow: scales
    # from 2^-126 there, and 2^128 and above is infinite
    e[:20] = rng.integers(-126 if dtype == "bfloat16" else -149, 128, size=(20, G))
    S = (rng.choice([-1.0, 1.0], size=(dout, G)) * rng.uniform(1, 2, size=(dout, G)) * 2.0 ** e).astype(np.float32)
    S[20:40] = (rng.integers(1, 1 << 12, size=(20, G)) * 2.0 ** -20).astype(np.float32)   # many ties
    S[40, :3] = [0.0, np.inf, -np.inf]
    Q = rng.integers(0, 256, size=(dout, din), dtype=np.uint8)
    Z = rng.integers(0, 256, size=(dout, G)).astype(np.int32)
    with np.errstate(over="ignore", invalid="ignore"):
        ref = np.asarray(dequantize_cast(S, Q, Z, g, dtype), dtype=np.float64)
    if dtype == "bfloat16":
        ref[np.abs(ref) >= 2.0 ** 128] *= np.inf
    t = lambda a: torch.as_tensor(a).cuda()
    out = jarq.dequantize(t(S), _offset_copy(Q, off), t(Z), g, bits, dtype).double().cpu().numpy()
    np.testing.assert_array_equal(out, ref)


@pytest.mark.parametrize("g,off", [(64, 0), (64, 1), (30, 0)])
def test_canonicalize_paths_agree(jarq, g, off):
    S, Q, Z = _signed_state(45, 5 * g, g, 4, seed=g)
    S2, Q2, Z2 = canonicalize(S.astype(np.float64), Q, Z, 4)
    Sd, Zd, Qd = torch.as_tensor(S).cuda(), torch.as_tensor(Z).cuda(), _offset_copy(Q, off)
    jarq.canonicalize(Sd, Qd, Zd, g, 4)
    assert np.array_equal(Sd.cpu().numpy(), S2.astype(np.float32))
    assert np.array_equal(Qd.cpu().numpy(), Q2) and np.array_equal(Zd.cpu().numpy(), Z2)


@pytest.mark.parametrize("bits", [1, 2, 3, 4, 5, 6, 7, 8])
@pytest.mark.parametrize("off", [0, 1])
def test_pack_codes_whole_words(jarq, bits, off):
    """Rows of a multiple of 32 codes: 32 codes a thread, or the general kernel
    for misaligned codes."""
    rng = np.random.default_rng(bits)
    Q = rng.integers(0, 1 << bits, size=(37, 96), dtype=np.uint8)
    got = jarq.pack_codes(_offset_copy(Q, off), bits).cpu().numpy().view(np.uint32)
    assert np.array_equal(got, pack_codes(Q, bits))


@pytest.mark.parametrize("bits", [2, 3, 4, 5, 6, 7, 8])
def test_pack_codes_bit_exact(jarq, bits):
    rng = np.random.default_rng(bits)
    Q = rng.integers(0, 1 << bits, size=(33, 203), dtype=np.uint8)    # ragged: 203 b not a multiple of 32
    ref = pack_codes(Q, bits)
    got = jarq.pack_codes(torch.as_tensor(Q).cuda(), bits).cpu().numpy().view(np.uint32)
    assert np.array_equal(got, ref)


def test_writeback_rejects_bad_input(jarq):
    S, Q, Z = _signed_state(8, 128, 64, 3, seed=1)
    lib = jarq.library()
    # host pointers
    assert lib.jarq_pack_codes(Q.ctypes.data, 8, 128, 3, Q.ctypes.data, None) == jarq.JARQ_ERR_ARG
    # a code outside [0, qmax] is rejected before any change
    Qd = torch.as_tensor(Q).cuda()
    Qd[3, 5] = 8
    Sd, Zd = torch.as_tensor(S).cuda(), torch.as_tensor(Z).cuda()
    S0 = Sd.clone()
    with pytest.raises(jarq.JarqError):
        jarq.canonicalize(Sd, Qd, Zd, 64, 3)
    assert torch.equal(Sd, S0)
    # the cast leaves its output alone as well
    Wd = torch.full((8, 128), 7.0, dtype=torch.float16, device="cuda")
    assert lib.jarq_dequantize(Sd.data_ptr(), Qd.data_ptr(), Zd.data_ptr(), 8, 128, 64, 3, 1,
                               Wd.data_ptr(), None) == jarq.JARQ_ERR_ARG
    assert bool((Wd == 7.0).all())


def test_valid_and_invalid_layers_on_two_streams(jarq):
    """Two host threads, each on a stream of its own, one writing back a valid
    layer and one passing codes out of range, over and over: every valid result
    is whole, every invalid call is refused and changes nothing."""
    import threading
    dout, din, g, bits = 1031, 2048, 64, 3
    S, Q, Z = _signed_state(dout, din, g, bits, seed=77)
    S2, Q2, Z2 = canonicalize(S.astype(np.float64), Q, Z, bits)
    want = {"S": S2.astype(np.float32), "Q": Q2, "Z": Z2, "P": pack_codes(Q2, bits).view(np.int32),
            "W": np.asarray(dequantize_cast(S2.astype(np.float32), Q2, Z2, g, "float16"), dtype=np.float16)}
    want = {k: torch.as_tensor(v).cuda() for k, v in want.items()}
    t = lambda a: torch.as_tensor(a).cuda()
    Sd, Qd, Zd = t(S), t(Q), t(Z)
    Qbad = Qd.clone()
    Qbad[-1, -1] = 1 << bits            # seen by the last blocks of the check
    torch.cuda.synchronize()
    wrong, done = [], threading.Event()

    def valid():
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                for _ in range(150):
                    s, q, z = Sd.clone(), Qd.clone(), Zd.clone()
                    jarq.canonicalize(s, q, z, g, bits)
                    got = {"S": s, "Q": q, "Z": z, "W": jarq.dequantize(s, q, z, g, bits, "float16"),
                           "P": jarq.pack_codes(q, bits)}
                    wrong.extend(k for k, v in got.items() if not torch.equal(v, want[k]))
        except Exception as e:      # a valid call refused
            wrong.append(e)
        done.set()

    def invalid():
        with torch.cuda.stream(torch.cuda.Stream()):
            s, q, z = Sd.clone(), Qbad.clone(), Zd.clone()
            while not done.is_set():
                for call in (lambda: jarq.canonicalize(s, q, z, g, bits), lambda: jarq.pack_codes(q, bits),
                             lambda: jarq.dequantize(s, q, z, g, bits, "float16")):
                    try:
                        call()
                        wrong.append("an invalid layer was accepted")
                    except jarq.JarqError as e:
                        if e.status != jarq.JARQ_ERR_ARG:
                            wrong.append(e)
            if not (torch.equal(s, Sd) and torch.equal(q, Qbad) and torch.equal(z, Zd)):
                wrong.append("an invalid layer was changed")

    threads = [threading.Thread(target=f) for f in (valid, invalid)]
    for th in threads:
        th.start()
    for th in threads:
        th.join(120)
    assert done.is_set() and not wrong, wrong[:5]


def test_ridge_acceptance_matches_oracle(jarq):
    """A row whose starting scales are its exact least-squares scales and
    whose Gram matrix is singular (one group at its zero point, H scaled so
    the ridge bias shows): the ridge solve raises F, so with the option the
    previous scales are kept, without it they are not (App. G Remark
    ridge-acceptance); codes and scales match the oracle either way."""
    lay = small_layer(256, 4, 64, 3, seed=5, rank=8, tokens=1200)
    H = (lay.H.astype(np.float64) * 1e-4).astype(np.float32)
    Q = lay.Q0.copy()
    Q[1, 64:128] = lay.Z[1, 1]
    prep = prepare_hessian(H, 64)
    Gram, rhs = scale_system(prep, lay.W[1:2], Q[1:2], lay.Z[1:2])
    keep = [0, 2, 3]
    S0 = lay.S0.astype(np.float32).copy()
    S0[1, keep] = np.linalg.solve(Gram[0][np.ix_(keep, keep)], rhs[0][keep]).astype(np.float32)
    for accept in (0, 1):
        res = refine_layer(prep, lay.W, S0, Q, lay.Z, 3,
                           Options(max_iters=1, early_stop=False, ridge_accept=bool(accept)))
        t = lambda a: torch.as_tensor(np.ascontiguousarray(a)).cuda()
        hess = jarq.prepare(t(H), 64)
        S, Qd = t(S0), t(Q)
        st = jarq.refine(hess, t(lay.W), S, Qd, t(lay.Z), 3, max_iters=1, early_stop=0,
                         ridge_accept=accept, raise_on_error=False)
        hess.close()
        Sg = S.cpu().numpy()
        assert int(st.ridge_hits.cpu()[1]) == 1
        assert np.array_equal(Qd.cpu().numpy(), res.Q)
        np.testing.assert_allclose(Sg, res.S, rtol=1e-6)
        if accept:
            assert np.array_equal(Sg[1], S0[1])
        else:
            assert not np.array_equal(Sg[1], S0[1])
