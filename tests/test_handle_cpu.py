"""Host side of a handle: errors at its making, the size of its workspace."""

import ctypes

import pytest

from paper_2503_10380_gb300 import binding


@pytest.fixture(scope="module")
def lib():
    import __graft_entry__
    try:
        __graft_entry__.build()
    except RuntimeError as e:   # no nvcc on this machine
        pytest.skip(str(e))
    return binding.lib()


def test_a_kernel_that_cannot_run_is_an_error(lib):
    """Where the FP64 contraction kernel cannot be set up (here: no GPU) a handle of any
    precision says so when it is made, instead of taking a slower kernel without a word."""
    torch = pytest.importorskip("torch")
    if torch.cuda.is_available():
        pytest.skip("needs a machine without a GPU: the pointers below are not real")
    opts = binding.make_opts("fp64")
    need = binding.ppl_cpd_workspace_size(5, 24, 72, 48, opts)
    h, fake = ctypes.c_void_p(), 1 << 20
    rc = lib.ppl_cpd_init(ctypes.byref(h), 5, 24, 72, 48, fake, fake, fake, fake, need, ctypes.byref(opts), None)
    assert rc == binding.PPL_ECUDA and not h
    assert b"FP64 contraction kernel" in lib.ppl_last_error(None)


# (o, v, X, R) -> bytes in FP64, BF16X3, TF32 dressed, TF32X3, TF32X3 with r_chunk 96
WORKSPACE = {
    (5, 24, 72, 48): (5606656, 10162432, 8776960, 10899712, 10899712),
    (10, 90, 270, 250): (426033408, 526692096, 537212160, 660349696, 548976896),
    (13, 117, 355, 331): (490484224, 755482112, 879183104, 1167324160, 872277248),
    (14, 120, 360, 160): (462711296, 595708416, 723790336, 862398976, 781246976),
    (20, 200, 600, 800): (1346521344, 3707353344, 4021926144, 6075250944, 3547404544),
    (60, 600, 1800, 2400): (29022668544, 71141017344, 84956415744, 120338482944, 99562546944),
    (1, 2, 3, 1): (22528, 35328, 32512, 35328, 35328),
}


@pytest.mark.parametrize("shape", WORKSPACE)
def test_workspace_does_not_grow(lib, shape):
    """A program with a fixed allocation for its handles keeps fitting: faster forms of a
    call find their scratch in what the handle has."""
    kinds = (("fp64", {}), ("bf16x3", {}), ("tf32", {"dressed": True}), ("tf32x3", {}), ("tf32x3", {"r_chunk": 96}))
    for (prec, kw), limit in zip(kinds, WORKSPACE[shape]):
        need = binding.ppl_cpd_workspace_size(*shape, binding.make_opts(prec, **kw))
        assert need <= limit, (prec, kw, need, limit)
