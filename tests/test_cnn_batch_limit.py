"""The network's forward counts a layer's rows, 1024 a patch in the first, in 32 bits: more patches than that holds are
refused before anything is launched (2^21 of them used to be taken for an empty first layer, and the call to
have succeeded).  The workspace is NULL, so that a call that passes this check launches nothing either and
says so (CELESTE_ERR_WORKSPACE)."""
import ctypes

import pytest

INVALID_ARG, WORKSPACE = 1, 4


@pytest.mark.parametrize("engine", [0, 1])
@pytest.mark.parametrize("batch,rc", [((1 << 21) - 1, WORKSPACE), (1 << 21, INVALID_ARG), ((1 << 31) - 1, INVALID_ARG)])
def test_batch_limit(batch, rc, engine):
    import __graft_entry__
    __graft_entry__.build()
    import paper_1611_03404_gb300 as P
    L = P.lib()
    a, none, size = ctypes.c_void_p(1 << 20), ctypes.c_void_p(0), ctypes.c_size_t(0)   # (a is never read)
    assert L.celeste_cnn_forward_ex(a, a, a, batch, none, none, a, none, size, engine, none) == rc
    if engine == 1:
        assert L.celeste_cnn_forward(a, a, a, batch, none, none, a, none, size, none) == rc
