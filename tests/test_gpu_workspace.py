"""What calls leave in a handle's workspace: the exact contractions and the reconstruction
use parts of it that belong to other calls, and no call may read what it did not write.

Every handle here gets a workspace full of NaN (0xff bytes).
"""

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2503_10380_gb300 import binding, inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()


class _Poisoned(binding.CpAls):
    """CpAls whose workspace held NaN before the handle was made"""

    def __init__(self, *a, **k):
        empty = torch.empty

        def poisoned(*s, **kw):
            t = empty(*s, **kw)
            return t.view(torch.uint8).fill_(255) if kw.get("dtype") == torch.uint8 else t

        torch.empty = poisoned
        try:
            super().__init__(*a, **k)
        finally:
            torch.empty = empty


# mixed exact contraction, rows a per launch: partials over the sweep's intermediates, behind
# G, one row only; a first size without K padding
SHAPES = [(8, 64, 41, 150), (8, 97, 41, 200), (8, 97, 41, 20), (2, 330, 8, 9), (3, 11, 17, 13)]


@pytest.mark.parametrize("prec", ["fp64", "bf16x3", "tf32", "tf32x3"])
@pytest.mark.parametrize("shape", SHAPES)
def test_calls_leave_the_workspace_to_each_other(prec, shape):
    o, v, X, R = shape
    inp = inputs.make_inputs(o, v, X, R, seed=11)
    dev = [torch.from_numpy(np.ascontiguousarray(x)).cuda() for x in (inp.B, inp.tau)]

    def mttkrps(cp):
        return [cp.mttkrp(m) for m in ("a", "b", "i", "j")]

    cp = _Poisoned(*dev, inp.factors, precision=prec, want_eta=True)
    first = mttkrps(cp)
    calls = {
        "reconstruct": lambda c: [c.reconstruct(symmetrise=True)],
        "energy": lambda c: [torch.tensor(c.energy())],
    }
    if v < 300:
        calls["exact"] = lambda c: [c.exact_contract(want_R=True)[2]]
    if prec != "fp64":
        calls["mixed"] = lambda c: [c.exact_contract(want_R=True, mixed=True)[2]]
        calls["mixed sums"] = lambda c: [torch.tensor(c.exact_contract(mixed=True)[:2])]
    alone = {}
    for name, call in calls.items():
        fresh = _Poisoned(*dev, inp.factors, precision=prec)
        alone[name] = call(fresh)
        fresh.close()
        assert all(bool(torch.isfinite(x).all()) for x in alone[name]), name
    # FP64 split-K sums are atomic: the last bits of an MTTKRP may differ from call to call
    same = torch.equal if prec != "fp64" else lambda a, b: torch.allclose(a, b, rtol=1e-12, atol=1e-13 * float(b.abs().max()))
    for order in (list(calls), list(calls)[::-1]):
        for name in order:
            for a, b in zip(calls[name](cp), alone[name]):
                assert torch.equal(a, b), (name, order)
            for a, b in zip(mttkrps(cp), first):
                assert bool(torch.isfinite(a).all()) and same(a, b), (name, order)
    cp.sweep(2)
    assert all(bool(torch.isfinite(x).all()) for x in cp.factors().values())
    cp.close()
