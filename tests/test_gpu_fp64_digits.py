"""FP64 contractions formed from exact digit products (csrc/ppl_split64.cu), against exact
integer arithmetic.

The reconstruction R~[a,b,i,j] = sum_r Ua[a,r] Ub[b,r] Ui[i,r] Uj[j,r] with U_b = U_j = 1
is one contraction of the rows of U_a with the rows of U_i over K = R, so any rows can
be tried:

* the digit form must be no worse than the FP64 FMA chain it stands for on any rows: the
  chain is evaluated exactly here, and over the 240 elements of a case the rms error (in
  units of the sum of the |terms|) may be 1.25 times the chain's and the largest error
  twice the chain's (what two samples of that size differ by).
* for sums without cancellation the digit form is rounded once: 0.51 units in the last
  place.  A chain of 256 FMAs is several units off, so this also shows which kernel ran.
"""

import math
import time
from fractions import Fraction

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import ppl_oracle as orc
from paper_2503_10380_gb300 import binding, inputs
from parity import abs_factors, check_abs_bound

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()


def _handle(A, B, precision="fp64", **opts):
    """A handle whose reconstruction is A B^T: A [v][K] in mode a, B [o][K] in mode i."""
    (v, K), o = A.shape, B.shape[0]
    fac = {"a": A, "b": np.ones((v, K)), "i": B, "j": np.ones((o, K))}
    g = torch.Generator().manual_seed(0)
    Bt = torch.randn(2, o + v, o + v, generator=g, dtype=torch.float64)
    tau = torch.randn(o, o, v, v, generator=g, dtype=torch.float64)
    return binding.CpAls((Bt + Bt.transpose(1, 2)).cuda(), tau.cuda(), fac, precision=precision, **opts)


def _products(A, B, precision="fp64"):
    """[v][o] from the device: of the copies [b][j] of an element, one from all over the output"""
    cp = _handle(A, B, precision)
    R = cp.reconstruct(symmetrise=False).cpu().numpy()       # [a][b][i][j]
    cp.close()
    a, i = np.meshgrid(np.arange(A.shape[0]), np.arange(B.shape[0]), indexing="ij")
    return R[a, (7 * a + 3 * i) % A.shape[0], i, (a + i) % B.shape[0]]


def _ints(A):
    """A = ints 2^-s, exactly"""
    low = min((math.frexp(x)[1] for x in A.ravel() if x != 0.0), default=0)
    s = 53 - low
    return np.array([[int(Fraction(float(x)) * Fraction(2) ** s) for x in r] for r in A], dtype=object), s


def _errors(got, A, B):
    """|got - exact| and sum |terms|, both as floats, and the exact values"""
    (IA, sa), (IB, sb) = _ints(A), _ints(B)
    unit = Fraction(2) ** -(sa + sb)
    ex = [[Fraction(int(x)) * unit for x in r] for r in IA @ IB.T]
    ab = np.array([[float(Fraction(int(x)) * unit) for x in r] for r in np.abs(IA) @ np.abs(IB).T])
    err = np.array([[float(abs(Fraction(float(g)) - e)) for g, e in zip(gr, er)] for gr, er in zip(got, ex)])
    return err, ab, np.array([[float(e) for e in r] for r in ex])


def _fma_chain(x, y):
    s = 0.0
    for p, q in zip(x, y):
        s = float(Fraction(float(p)) * Fraction(float(q)) + Fraction(s))     # rounded once
    return s


def _rows(kind, K, rng, v=40, o=6):
    A, B = rng.standard_normal((v, K)), rng.standard_normal((o, K))
    if kind.startswith("opposed"):                # one operand large where the other is small
        s = 2.0 ** -int(kind[7:])
        A[:, K // 2:] *= s
        B[:, :K // 2] *= s
    elif kind.startswith("spread"):
        s = float(kind[6:])
        A *= 2.0 ** rng.uniform(-s, 0, A.shape)
        B *= 2.0 ** rng.uniform(-s, 0, B.shape)
    elif kind == "decay":
        d = np.exp(-np.arange(K) / 15.0)
        A *= d
        B *= d
    return A, B


@pytest.mark.parametrize("kind,K", [("even", 8), ("even", 33), ("opposed3", 8), ("opposed5", 8), ("opposed7", 8),
                                    ("opposed10", 9), ("opposed6", 64), ("opposed9", 64), ("spread16", 32),
                                    ("spread24", 128), ("decay", 150), ("spread40", 40),
                                    ("spread24", 300)])
def test_no_worse_than_an_fma_chain(kind, K):
    A, B = _rows(kind, K, np.random.default_rng(K))
    err, ab, _ = _errors(_products(A, B), A, B)
    chain, _, _ = _errors([[_fma_chain(x, y) for y in B] for x in A], A, B)
    r, c = err / ab, chain / ab
    assert r.max() <= 2.0 * c.max(), (r.max(), c.max())
    assert np.sqrt(np.mean(r * r)) <= 1.25 * np.sqrt(np.mean(c * c))


@pytest.mark.parametrize("K", [8, 31, 32, 33, 128, 129, 256])
def test_sums_of_one_sign_are_rounded_once(K):
    rng = np.random.default_rng(100 + K)
    A, B = 0.5 + 0.5 * rng.random((40, K)), 0.5 + 0.5 * rng.random((6, K))
    err, _, ex = _errors(_products(A, B), A, B)
    assert np.max(err / np.spacing(ex)) <= 0.51


def test_largest_digits():
    """Every digit +127 or -128 over two full folds of 128 k: the FP32 sums of products of
    one weight come within an eighth of 2^24, and stay exact."""
    plus = 0x7f7f7f7f7f7f
    minus = 127 * 256 ** 5 - 128 * sum(256 ** k for k in range(5))
    K = 256
    A = np.array([[float(plus)] * K, [float(minus)] * K, [float(-minus)] * K, [float(plus), float(minus)] * (K // 2)])
    B = np.array([[float(minus)] * K, [float(plus)] * K])
    err, ab, ex = _errors(_products(A, B), A, B)
    assert np.all(err <= 0.51 * np.spacing(np.abs(ex)))


def test_largest_digits_over_many_folds():
    """The same with K = o^2 = 576: T[r][c][d] = sum_ij U_i[i][r] U_j[j][r] tau[i][j][c][d], which the
    MTTKRP of mode a passes on unchanged where B is the identity and U_b picks d = 0."""
    o, v, X, R = 24, 17, 2, 9
    plus = 0x7f7f7f7f7f7f
    minus = 127 * 256 ** 5 - 128 * sum(256 ** k for k in range(5))
    rows, cols = [plus, minus, -plus], [minus, plus, -minus, -plus]
    B = np.zeros((X, o + v, o + v))
    B[0, o:, o:] = np.eye(v)
    tau = np.broadcast_to(np.array([float(cols[c % 4]) for c in range(v)])[:, None], (o, o, v, v))
    fac = {"a": np.ones((v, R)), "b": np.zeros((v, R)), "j": np.ones((o, R)),
           "i": np.broadcast_to(np.array([float(rows[r % 3]) for r in range(R)]), (o, R))}
    fac["b"][0] = 1.0
    cp = binding.CpAls(torch.from_numpy(B).cuda(), torch.from_numpy(tau.copy()).cuda(),
                       {m: x.copy() for m, x in fac.items()}, precision="fp64")
    M = cp.mttkrp("a").cpu().numpy()
    cp.close()
    for c in range(v):
        for r in range(R):
            exact = o * o * rows[r % 3] * cols[c % 4]
            assert abs(int(M[c, r]) - exact) <= 0.51 * np.spacing(abs(float(exact))), (c, r)


@pytest.mark.parametrize("kind", ["random", "halves", "one", "wide"])
@pytest.mark.parametrize("K", [33, 200, 300])
def test_rows_with_zeros(kind, K):
    """Rows with few non-zero entries: a sum without a non-zero term is exactly zero, the
    others are as accurate as an FMA chain.  "wide": among the entries are some 2^-70 times
    the others, which the digits cannot hold."""
    rng = np.random.default_rng(7 * K + len(kind))
    A, B = rng.standard_normal((40, K)), rng.standard_normal((6, K))
    if kind == "halves":                 # supports of symmetry blocks
        A[::2, K // 2:] = 0.0
        A[1::2, :K // 2] = -0.0
        B[::2, K // 2:] = 0.0
        B[1::2, :K // 2] = 0.0
    elif kind == "one":
        A *= np.arange(K)[None] % 20 == np.arange(40)[:, None] % 20
        B *= np.arange(K)[None] % 20 == np.arange(6)[:, None]
    else:
        A *= rng.random(A.shape) < 0.1
        B *= rng.random(B.shape) < 0.1
        if kind == "wide":
            A *= np.where(rng.random(A.shape) < 0.5, 2.0 ** -70, 1.0)
    got = _products(A, B)
    err, ab, _ = _errors(got, A, B)
    assert np.all(got[ab == 0.0] == 0.0) and np.any(ab == 0.0) and np.any(ab > 0.0)
    chain, _, _ = _errors([[_fma_chain(x, y) for y in B] for x in A], A, B)
    r, c = err[ab > 0] / ab[ab > 0], chain[ab > 0] / ab[ab > 0]
    assert r.max() <= max(2.0 * c.max(), 2.0 ** -52)      # (few terms: an element is off by one rounding or two)


def test_cost_of_rows_with_zeros():
    """Nine in ten entries zero: a tenth of the elements is left to FP64 FMAs, the sums
    without a term are not.  Within six times the time of full rows (all tiles by FMAs
    take ten times and more)."""
    v, o, K = 150, 12, 400
    rng = np.random.default_rng(2)
    ms = []
    for density in (1.1, 0.1):
        A, B = rng.standard_normal((v, K)), rng.standard_normal((o, K))
        cp = _handle(A * (rng.random(A.shape) < density), B * (rng.random(B.shape) < density))
        best = math.inf
        for _ in range(8):
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            e0.record()
            cp.reconstruct(symmetrise=False)
            e1.record()
            torch.cuda.synchronize()
            best = min(best, e0.elapsed_time(e1))
        ms.append(best)
        cp.close()
    assert ms[1] <= 6.0 * ms[0], ms


@pytest.mark.parametrize("precision", ["fp64", "tf32x3"])
@pytest.mark.parametrize("K", [24, 300])
def test_wait_limit_holds(precision, K):
    """A wait that runs out (the first stage of one block never fills): the call reports
    PPL_ETIMEOUT after the handle's limit of 20 ms, not the default of 500, the other
    blocks' results stand aside, and the next call is right again."""
    rng = np.random.default_rng(5)
    A, B = 0.5 + rng.random((40, K)), 0.5 + rng.random((6, K))
    cp = _handle(A, B, precision, wait_limit_us=20000)
    before = cp.reconstruct(symmetrise=False)
    binding.ppl_cpd_inject_contraction_timeout(cp.h)
    t0 = time.perf_counter()
    with pytest.raises(binding.PplError) as e:
        cp.reconstruct(symmetrise=False)
    elapsed = time.perf_counter() - t0
    assert e.value.code == binding.PPL_ETIMEOUT, str(e.value)
    assert 0.015 < elapsed < 0.4, elapsed
    assert cp.stats()["timeouts"] == 1
    assert torch.equal(cp.reconstruct(symmetrise=False), before)
    assert cp.stats()["timeouts"] == 1
    cp.close()


def test_wait_limit_holds_in_a_captured_sweep():
    rng = np.random.default_rng(6)
    fac = {m: rng.standard_normal((24 if m in "ab" else 5, 16)) for m in "abij"}
    cp = _handle(fac["a"], fac["i"], wait_limit_us=20000)
    cp.set_factors(fac)
    cp.sweep(1)                          # captured; the flag is read at run time
    first = {m: x.clone() for m, x in cp.factors().items()}
    cp.set_factors(fac)
    binding.ppl_cpd_inject_contraction_timeout(cp.h)
    with pytest.raises(binding.PplError) as e:
        cp.sweep(1)
    assert e.value.code == binding.PPL_ETIMEOUT, str(e.value)
    cp.set_factors(fac)
    cp.sweep(1)
    for m, x in cp.factors().items():
        assert torch.allclose(x, first[m], rtol=1e-9, atol=1e-9 * float(first[m].abs().max()))
    assert cp.stats()["timeouts"] == 1
    cp.close()


@pytest.mark.parametrize("kind", ["zeros", "spread", "wide"])
@pytest.mark.parametrize("shape", [(5, 24, 72, 48), (3, 33, 97, 9), (9, 40, 150, 130)])
def test_every_layout_of_the_method(shape, kind):
    """MTTKRPs, the exact contraction and the energy in FP64 on inputs that leave elements to
    FP64 FMAs or have sums without terms, in each of the layouts the method contracts
    (strided and compound k, split K with atomic sums, batches).  "zeros": nine in ten
    entries of B and tau; "spread": auxiliary functions over 2^40, factors over 2^10;
    "wide": the entries of B over 2^60.  Bound: 1e-12 of the same chain on absolute values
    (four contractions of up to 6000 terms at 2^-53 each side)."""
    o, v, X, R = shape
    inp = inputs.make_inputs(o, v, X, R, seed=21)
    rng = np.random.default_rng(3)
    B, tau, U = inp.B.copy(), inp.tau.copy(), {m: x.copy() for m, x in inp.factors.items()}
    if kind == "zeros":
        mask = rng.random(B.shape) < 0.1
        B *= mask | mask.transpose(0, 2, 1)
        tau *= rng.random(tau.shape) < 0.1
    elif kind == "spread":
        B *= 2.0 ** rng.permutation(np.linspace(-20, 20, X))[:, None, None]
        for m in U:
            U[m] *= 2.0 ** rng.uniform(-5, 5, U[m].shape)
    else:
        s = rng.uniform(-30, 30, B.shape)
        B *= 2.0 ** (0.5 * (s + s.transpose(0, 2, 1)))
    Bvv, aB, at, aU = B[:, o:, o:], np.abs(B), np.abs(tau), abs_factors(U)
    cp = binding.CpAls(torch.from_numpy(B).cuda(), torch.from_numpy(tau).cuda(), U, precision="fp64")
    for m in orc.MODES:
        check_abs_bound(cp.mttkrp(m).cpu().numpy(), orc.mttkrp(Bvv, tau, U, m), orc.mttkrp(aB[:, o:, o:], at, aU, m), 1e-12,
                        f"{kind} {shape} mode {m}")
    n2, E, Rt = cp.exact_contract(want_R=True)
    check_abs_bound(Rt.cpu().numpy(), orc.ppl_tensor(Bvv, tau), orc.ppl_tensor(aB[:, o:, o:], at), 1e-12, f"{kind} {shape} R")
    one = np.ones(R)
    # with |a| + |b| in both virtual modes the direct and the exchange sum are alike, each at
    # least the sum of the |terms| of either; their difference 2 x - x is x
    scale = 3.0 * orc.energy_cp(aB, o, {**aU, "a": aU["a"] + aU["b"], "b": aU["a"] + aU["b"]}, one)
    assert abs(cp.energy() - orc.energy_cp(B, o, U, one)) <= 1e-12 * scale
    cp.close()
