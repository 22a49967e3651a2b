"""The counting kernels' grid follows the device of each launch: never more
blocks than that device's context has scratch regions for."""
import ctypes

import pytest

import paper_2403_01261_gb300 as gsl


class DeviceInfo(ctypes.Structure):
    _fields_ = [("sm_count", ctypes.c_int), ("max_smem_optin", ctypes.c_int), ("cooperative", ctypes.c_int)]


@pytest.mark.parametrize("per_sm", [0, 1, 4, 8, 32])
def test_no_more_blocks_than_scratch_regions(per_sm):
    lib = gsl.load()
    grid = lib._ZN3gsl11sketch_gridEibRKNS_10DeviceInfoE      # gsl::sketch_grid
    regions = lib._ZN3gsl13sketch_blocksERKNS_10DeviceInfoE   # gsl::sketch_blocks
    grid.restype, regions.restype = ctypes.c_int, ctypes.c_longlong
    grid.argtypes = [ctypes.c_int, ctypes.c_bool, ctypes.POINTER(DeviceInfo)]
    regions.argtypes = [ctypes.POINTER(DeviceInfo)]
    for sms in (152, 20, 152, 1):   # one host thread going from device to device
        di = DeviceInfo(sms, 232448, 1)
        assert grid(per_sm, True, di) == min(max(per_sm, 1) * sms, regions(di))
        assert grid(per_sm, False, di) == max(per_sm, 1) * sms
