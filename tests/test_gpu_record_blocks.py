"""argus_aggregate chooses between blocks of three sizes by how many of each the chip holds at once: what it takes for that is what the device says."""
import ctypes

import pytest

import paper_2609_12299_b200 as argus

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("threads", [256, 192, 128])
def test_blocks_an_sm_holds(threads):
    lib, rule, device = argus.load_library(), ctypes.c_uint32(), ctypes.c_uint32()
    for regions in range(1, 401):
        assert lib.argus_testing_record_blocks(regions, threads, ctypes.byref(rule), ctypes.byref(device)) == 0
        assert rule.value == device.value > 0, regions
