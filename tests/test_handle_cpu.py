"""Host side of a handle: errors at its making."""

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
