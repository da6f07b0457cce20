"""Rules of the dispatch that need no GPU: which kernel takes a cross-scan or
cross-merge of long rows, when the channel-mean scan takes two steps per thread, and
when the selection kernel takes two operand buffers."""
import ctypes

import pytest

F32, BF16 = 0, 1
PLANE, BAND, GATHER = 0, 1, 2
SMS = 152


@pytest.fixture(scope="module")
def lib():
    from paper_2412_16602_gb300 import _build
    lib = ctypes.CDLL(_build.build())
    i, ll = ctypes.c_int, ctypes.c_longlong
    lib.vmb_testing_csm_kernel.argtypes = [i, i, ll, i, i, i, i]
    lib.vmb_testing_mean_two_steps.argtypes = [ll, i, ll, ll, i, i]
    lib.vmb_testing_selection_buffers.argtypes = [ll, i, i]
    return lib


@pytest.mark.parametrize("merge,dt,H,W,aligned,kernel", [
    (0, F32, 31, 33, 1, PLANE), (1, BF16, 1, 1023, 0, PLANE),
    (0, F32, 32, 32, 1, BAND), (1, F32, 56, 56, 1, BAND),
    # rows too long for a band: whole planes while they fit shared memory
    (0, F32, 1, 9000, 1, PLANE), (0, F32, 8, 6000, 1, PLANE), (1, F32, 2, 8000, 1, PLANE), (0, BF16, 8, 8793, 1, PLANE),
    (0, F32, 8, 6000, 0, PLANE), (0, F32, 7, 6418, 1, PLANE), (0, F32, 3, 6803, 1, PLANE), (1, F32, 3, 3297, 1, GATHER),
    (0, BF16, 3, 8349, 1, PLANE), (0, F32, 9, 6000, 1, GATHER), (1, F32, 1, 9001, 1, GATHER),
    (0, F32, 16, 4000, 1, GATHER), (1, F32, 4, 6000, 1, GATHER), (1, BF16, 16, 7000, 1, GATHER),
    # planes larger than shared memory: bands where several share an SM
    (1, F32, 256, 256, 1, BAND), (1, F32, 64, 800, 1, GATHER), (1, F32, 512, 512, 1, GATHER),
    (1, F32, 201, 201, 1, GATHER), (1, F32, 256, 256, 0, GATHER), (1, F32, 14, 1948, 0, GATHER),
    (1, BF16, 128, 800, 1, BAND), (1, BF16, 401, 399, 1, BAND), (1, BF16, 7001, 12, 1, GATHER),
    (1, BF16, 61, 997, 1, GATHER), (0, F32, 128, 800, 1, BAND), (0, F32, 61, 997, 1, BAND), (0, F32, 19, 2999, 1, GATHER),
])
def test_csm_kernel(lib, merge, dt, H, W, aligned, kernel):
    assert lib.vmb_testing_csm_kernel(merge, dt, 192, H, W, aligned, SMS) == kernel


def test_csm_kernel_of_few_planes(lib):
    assert lib.vmb_testing_csm_kernel(1, F32, 16, 2, 8000, 1, SMS) == GATHER
    assert lib.vmb_testing_csm_kernel(0, F32, 6, 4, 7336, 1, SMS) == GATHER
    assert lib.vmb_testing_csm_kernel(0, F32, 32, 3, 3297, 1, SMS) == GATHER
    assert lib.vmb_testing_csm_kernel(0, F32, 76, 3, 3297, 1, SMS) == PLANE
    assert lib.vmb_testing_csm_kernel(0, F32, 19, 4, 4096, 1, SMS) == PLANE
    assert lib.vmb_testing_csm_kernel(0, F32, 18, 4, 4096, 1, SMS) == GATHER
    assert lib.vmb_testing_csm_kernel(1, BF16, 16, 7001, 12, 1, SMS) == BAND


def test_csm_kernel_of_the_largest_problems(lib):
    assert lib.vmb_testing_csm_kernel(0, F32, 1 << 31, 4, 4, 1, SMS) == GATHER
    assert lib.vmb_testing_csm_kernel(0, F32, 1, 1 << 15, 1 << 15, 1, SMS) == GATHER


@pytest.mark.parametrize("ctas,with_y,two", [
    (1, 0, 0), (304, 0, 0), (416, 0, 0), (416, 1, 0), (432, 1, 0), (456, 1, 0),  # at most one wave with one step
    (457, 1, 1), (560, 1, 1), (560, 0, 1), (608, 1, 1),                         # one wave with two, two with one
    (896, 1, 0), (624, 1, 0), (624, 0, 1), (1344, 0, 1),
    (4096, 0, 1), (4992, 1, 1), (12800, 0, 1), (12800, 1, 1),
])
def test_mean_two_steps(lib, ctas, with_y, two):
    assert lib.vmb_testing_mean_two_steps(ctas, 192, 3 * SMS, 4 * SMS, SMS, with_y) == two


def test_mean_two_steps_of_few_channels(lib):
    assert lib.vmb_testing_mean_two_steps(420, 7, 3 * SMS, 4 * SMS, SMS, 0) == 1
    assert lib.vmb_testing_mean_two_steps(216, 32, 3 * SMS, 4 * SMS, SMS, 1) == 0


def test_mean_two_steps_without_a_kernel(lib):
    assert lib.vmb_testing_mean_two_steps(4096, 192, 3 * SMS, 0, SMS, 0) == 0
    assert lib.vmb_testing_mean_two_steps(4096, 192, 0, 4 * SMS, SMS, 0) == 0


@pytest.mark.parametrize("grid,D,buffers", [(256, 768, 2), (304, 33, 2), (305, 768, 1), (38, 27, 1), (300, 32, 1)])
def test_selection_buffers(lib, grid, D, buffers):
    assert lib.vmb_testing_selection_buffers(grid, D, SMS) == buffers
