"""The clamped solve on several 32-wide blocks, and the split-K reduction's two ways of
widening its partial sums."""

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import ppl_oracle as orc
from paper_2503_10380_gb300 import binding, inputs
from parity import GAMMA, abs_factors, check_abs_bound

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()


def _dev(x):
    return torch.from_numpy(np.ascontiguousarray(x)).cuda()


def test_clamped_solve_of_six_blocks():
    """R = 161: V of mode a (and b) has rank 160, its last pivot, in the sixth block of one
    column, is rounding noise and is clamped where it is not above the tolerance (which of
    the two noises are, rounding decides).  With V' = L L^T the factored matrix, V' - V is at
    most a few times 2^-52 R max V_kk, so some scales l make U_a diag(l) V = M within a few
    hundred times that (the oracle's own sweep: 2e-14 of the largest |M|); mode j, last and
    regular, likewise."""
    o, v, X, R = 4, 10, 12, 161
    inp = inputs.make_inputs(o, v, X, R, seed=13)
    cp = binding.CpAls(_dev(inp.B), _dev(inp.tau), inp.factors, precision="fp64")
    cp.sweep(1)
    f = {m: x.cpu().numpy() for m, x in cp.factors().items()}
    assert cp.stats()["clamped_pivots"] >= 1
    cp.close()

    def gram(U, modes):
        return np.prod([U[m].T @ U[m] for m in modes], axis=0)

    M, V = orc.mttkrp(inp.Bvv, inp.tau, inp.factors, "a"), gram(inp.factors, "bij")
    # U diag(l) V = M, linear in l
    lhs = (f["a"][:, None, :] * V.T[None]).reshape(v * R, R)
    l = np.linalg.lstsq(lhs, M.reshape(-1), rcond=None)[0]
    assert np.max(np.abs(lhs @ l - M.reshape(-1))) <= 1e-11 * np.max(np.abs(M))
    M, V = orc.mttkrp(inp.Bvv, inp.tau, f, "j"), gram(f, "abi")
    assert np.max(np.abs((f["j"] * f["lam"]) @ V - M)) <= 1e-11 * np.max(np.abs(M))


def _mode_a(B, inp, prec="tf32x3"):
    cp = binding.CpAls(_dev(B), _dev(inp.tau), inp.factors, precision=prec)
    M = cp.mttkrp("a").cpu().numpy()
    cp.close()
    return M


@pytest.mark.parametrize("few", [2, 6])
def test_subnormal_partial_sums(few):
    """Auxiliary functions of 2^-58 next to ones of 2^-66, whose slices' partial sums (the
    product of two, 2^-132) are subnormal in FP32: most of the slices, with two or six
    normal ones among them.  Subnormals are exact to 2^-149 each; read as if they were
    normal they would be 2^-127 and more."""
    inp = inputs.make_inputs(5, 24, 72, 48, seed=4)
    scale = np.full(72, 2.0 ** -66)
    scale[np.random.default_rng(1).permutation(72)[:few]] = 2.0 ** -58
    B = inp.B * np.exp(np.arange(72) / 15.0)[:, None, None] * scale[:, None, None]      # (no decay along Q)
    Bvv = B[:, 5:, 5:]
    ref = orc.mttkrp(Bvv, inp.tau, inp.factors, "a")
    ref_abs = orc.mttkrp(np.abs(Bvv), np.abs(inp.tau), abs_factors(inp.factors), "a")
    got = _mode_a(B, inp)
    # in units of 2^-116, the last bits of 72 slices (below) on top
    s = 2.0 ** 116
    check_abs_bound(got * s, ref * s, ref_abs * s + 72 * 24 * 2.0 ** -33 / GAMMA["tf32x3"], GAMMA["tf32x3"], f"{few} normal")


def test_all_partial_sums_subnormal():
    """Every partial sum subnormal: 72 slices, each the sum of at most two restarted chunks of
    twelve MMAs that end at 2^-149."""
    inp = inputs.make_inputs(5, 24, 72, 48, seed=4)
    B = inp.B * np.exp(np.arange(72) / 15.0)[:, None, None] * 2.0 ** -66
    ref = orc.mttkrp(B[:, 5:, 5:], inp.tau, inp.factors, "a")
    ref_abs = orc.mttkrp(np.abs(B[:, 5:, 5:]), np.abs(inp.tau), abs_factors(inp.factors), "a")
    assert 2.0 ** -132 < np.max(np.abs(ref)) < 2.0 ** -126
    err = np.abs(_mode_a(B, inp) - ref)
    assert np.all(err <= 72 * 24 * 2.0 ** -149 + GAMMA["tf32x3"] * ref_abs), np.max(err) * 2.0 ** 149


@pytest.mark.parametrize("x", [np.nan, np.inf])
def test_partial_sums_that_are_not_finite(x):
    """One entry of one auxiliary function: its slice makes every element of mode a not
    finite, whatever the others hold, and no other handle sees any of it."""
    inp = inputs.make_inputs(5, 24, 72, 48, seed=4)
    B = inp.B.copy()
    B[40, 7, 9] = B[40, 9, 7] = x
    assert not np.any(np.isfinite(_mode_a(B, inp)))
    assert np.all(np.isfinite(_mode_a(inp.B, inp)))
