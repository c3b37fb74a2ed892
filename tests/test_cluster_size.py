"""The size of a kernel's cluster launches is kept only when the device gave
it: a failed query (here: no device, or a pointer that is no kernel) must not
leave the process at one block."""
import ctypes as C

from paper_1705_02313_gb300 import build


def test_failed_queries_are_not_kept():
    lib = C.CDLL(build.build())
    ask = lib._ZN2pg14cluster_blocksEPKvimiiPSt6atomicIiE
    ask.argtypes = [C.c_void_p, C.c_int, C.c_size_t, C.c_int, C.c_int, C.c_void_p]
    ask.restype = C.c_int
    no_kernel = C.create_string_buffer(64)
    for shared in (0, 1 << 17):
        for device in (0, 63, 64, -1):
            cache = (C.c_int * 64)()
            assert ask(C.cast(no_kernel, C.c_void_p), 1024, shared, 16, device, cache) == 1
            assert not any(cache), (shared, device)
