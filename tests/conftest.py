import os
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)


def pytest_configure(config):
    config.addinivalue_line("markers", "gpu: needs a CUDA GPU (GB300, sm_103a)")
    config.addinivalue_line("markers", "slow: large CPU-side case")


@pytest.fixture(scope="session")
def polyq_lib():
    """The C-ABI library, built in-tree on first use."""
    from paper_2607_14618_gb300 import build as _build
    _build.build_library()
    from paper_2607_14618_gb300 import polyq
    return polyq


@pytest.fixture(scope="session")
def polyq_debug(polyq_lib):
    """The debug build of the library (include/polyq_debug*.h), by ctypes."""
    import ctypes as C

    from paper_2607_14618_gb300 import build
    lib = C.CDLL(build.build_library(debug=True))
    P, L = C.c_void_p, C.POINTER(polyq_lib.DevLayer)
    lib.polyq_debug_gemv_codes.argtypes = [L, P, C.c_int, P, P, C.c_size_t, P, P]
    lib.polyq_debug_gemm_weights.argtypes = [L, P, C.c_int64, P, P, C.c_size_t, P, P]
    lib.polyq_debug_linear_gemm.argtypes = [L, P, C.c_int64, P, P, C.c_size_t, C.c_int, P, P]

    class Choice(C.Structure):
        _fields_ = [("tokens", C.c_int32), ("pairs", C.c_int32), ("ksplit", C.c_int32),
                    ("streamk", C.c_int32), ("whole", C.c_int64)]

    lib.polyq_debug_gemm_choice.argtypes = [L, C.c_int64, C.POINTER(Choice)]
    lib.polyq_last_error.restype = C.c_char_p

    def gemm_choice(dev, M):
        """What polyq_linear_gemm launches for M tokens of the device layer."""
        c = Choice()
        assert lib.polyq_debug_gemm_choice(C.byref(dev.desc), M, C.byref(c)) == 0, \
            lib.polyq_last_error()
        return c

    lib.gemm_choice = gemm_choice
    return lib
