import os
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)


def pytest_configure(config):
    config.addinivalue_line("markers", "gpu: needs a CUDA GPU (GB300, sm_103a) and the built library")
    config.addinivalue_line("markers", "slow: long-running on CPU")


@pytest.fixture
def full_plan():
    """(tile shape, L-chunks, launched early) that the planner picks for a full scan
    (needs a GPU); `off`: u or x (1), delta (2) one element past 16-byte alignment."""
    import ctypes

    import paper_2412_16602_gb300 as vmb

    i = ctypes.c_int
    vmb.lib.vmb_testing_full_plan.argtypes = [i] * 6 + [ctypes.c_uint, i, i, i, ctypes.c_void_p]

    def plan(B, K, D, N, H, W, dt, map=False, off=0, flags=vmb.VMB_FLAG_SOFTPLUS):
        out = (i * 3)()
        s = vmb.lib.vmb_testing_full_plan(B, K, D, N, H, W, flags, vmb.VMB_F32 if dt == "f32" else vmb.VMB_BF16, int(map),
                                          off, out)
        assert s == vmb.VMB_OK
        return tuple(out)

    return plan


@pytest.fixture
def force_plan():
    """Force a tile shape / chunk count of the full scan ("shape[,chunks]") or a
    chunk length or the steps per thread of the channel-mean scan, or let the
    encoding of tensor maps fail, through libvmb's test-only controls
    (declared in paper_2412_16602_gb300/csrc/vmb_testing.h, not in the public
    header); the planners are restored when the test ends."""
    import ctypes
    import types

    import paper_2412_16602_gb300 as vmb

    lib = vmb.lib
    lib.vmb_testing_force_full_plan.argtypes = [ctypes.c_int, ctypes.c_int]
    lib.vmb_testing_force_full_plan.restype = ctypes.c_int
    lib.vmb_testing_force_mean_chunk.argtypes = [ctypes.c_int]
    lib.vmb_testing_force_mean_chunk.restype = ctypes.c_int
    lib.vmb_testing_force_mean_steps.argtypes = [ctypes.c_int]
    lib.vmb_testing_refuse_tensor_maps.argtypes = [ctypes.c_int]

    def full(spec: str):
        shape, _, chunks = str(spec).partition(",")
        assert lib.vmb_testing_force_full_plan(int(shape), int(chunks or 0)) == 0

    def mean(tc):
        assert lib.vmb_testing_force_mean_chunk(int(tc)) == 0

    def mean_steps(n):
        assert lib.vmb_testing_force_mean_steps(int(n)) == 0

    def refuse_tensor_maps(on=True):
        assert lib.vmb_testing_refuse_tensor_maps(int(on)) == 0

    try:
        yield types.SimpleNamespace(full=full, mean=mean, mean_steps=mean_steps, refuse_tensor_maps=refuse_tensor_maps)
    finally:
        lib.vmb_testing_force_mean_steps(0)
        lib.vmb_testing_refuse_tensor_maps(0)
        lib.vmb_testing_force_full_plan(-1, 0)
        lib.vmb_testing_force_mean_chunk(0)
