"""Host checks of the network's entry points that need no GPU: BF16 weights off a 16-byte boundary are refused
by the tcgen05 forward before anything is launched (its 16-byte copies would fault), and by no other
check.  The workspace is NULL throughout, so that a call that passes the checks under test launches nothing
either and says so (CELESTE_ERR_WORKSPACE)."""
import ctypes

import pytest

INVALID_ARG, WORKSPACE = 1, 4


@pytest.mark.parametrize("shift,forward", [(0, WORKSPACE), (2, INVALID_ARG), (8, INVALID_ARG), (14, INVALID_ARG)])
def test_weight_alignment(shift, forward):
    import __graft_entry__
    __graft_entry__.build()
    import paper_1611_03404_gb300 as P
    L = P.lib()
    a = lambda off=0: ctypes.c_void_p((1 << 20) + off)   # (never read)
    w, none = a(shift), ctypes.c_void_p(0)
    size, budget = ctypes.c_size_t(0), ctypes.c_longlong(0)
    assert L.celeste_cnn_forward(a(), w, a(), 1, none, none, a(), none, size, none) == forward
    assert L.celeste_cnn_forward_ex(a(), w, a(), 1, none, none, a(), none, size, 1, none) == forward
    assert L.celeste_cnn_forward_budget(a(), w, a(), 1, none, none, a(), none, size, 1, budget, none) == forward
    # the other engine and the backward pass take the weights anywhere
    assert L.celeste_cnn_forward_ex(a(), w, a(), 1, none, none, a(), none, size, 0, none) == WORKSPACE
    assert L.celeste_cnn_backward(a(), w, a(), a(), 1, a(), none, size, none) == WORKSPACE
