"""Plan.host_ptr is a ctypes pointer, so that it passes whole to a foreign function without argument types
(a plain integer would be cut to 32 bits there)."""
import ctypes

from paper_1310_7114_gb300 import itc


def test_host_ptr_is_a_pointer():
    plan = itc.Plan.__new__(itc.Plan)
    plan.host = ctypes.create_string_buffer(b"plan bytes", 64)
    p = plan.host_ptr
    assert isinstance(p, ctypes.c_void_p) and p.value == ctypes.addressof(plan.host)
    strlen = ctypes.CDLL(None).strlen   # no argument types
    strlen.restype = ctypes.c_size_t
    assert strlen(p) == 10
