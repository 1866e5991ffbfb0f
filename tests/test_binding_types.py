"""The C library through ctypes: tn_serve_submit_batch takes its array of input arrays in either form, an array
of pointers to pointers or of plain addresses (a null server is refused after the arguments are)."""
import ctypes as C

from tests._lib import ensure_built


def test_submit_batch_argument_forms():
    tn = ensure_built()
    from paper_2606_01852_gb300.binding import lib
    plans, leaves, tickets = (C.c_void_p * 1)(), (C.c_void_p * 2)(), (C.c_uint64 * 1)()
    pointers = (C.POINTER(C.c_void_p) * 1)(C.cast(leaves, C.POINTER(C.c_void_p)))
    addresses = (C.c_void_p * 1)(C.addressof(leaves))
    for inputs in (pointers, addresses, C.cast(pointers, C.POINTER(C.POINTER(C.c_void_p)))):
        assert lib.tn_serve_submit_batch(None, 1, plans, inputs, tickets) == tn.TN_ERR_INVALID
