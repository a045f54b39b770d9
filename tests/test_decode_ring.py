"""The ring of the decode kernel: how deep it is for every head layout, cluster size and amount of shared memory.  Host code, no GPU."""
import ctypes as C

import pytest

from paper_2502_05431_b200 import build as ape_build
from paper_2502_05431_b200 import libape

OPTIN, GROUPS = 232448 - 2048, 2        # what a plan gives the kernel of the 227 KB of a block; groups of warps that take turns at the tiles


@pytest.fixture(scope="module")
def lib():
    ape_build.build()
    lib = libape.load()
    lib.pick = getattr(lib, "_ZN3ape18decode_pick_stagesEiimi")       # ape::decode_pick_stages(int, int, size_t, int)
    lib.size = getattr(lib, "_ZN3ape17decode_smem_bytesEiiii")        # ape::decode_smem_bytes(int, int, int, int)
    lib.pick.argtypes, lib.pick.restype = [C.c_int, C.c_int, C.c_size_t, C.c_int], C.c_int
    lib.size.argtypes, lib.size.restype = [C.c_int, C.c_int, C.c_int, C.c_int], C.c_size_t
    return lib


@pytest.mark.parametrize("D", [64, 128])
@pytest.mark.parametrize("G", [1, 2, 4, 8, 16])
def test_a_stage_always_belongs_to_the_same_group(lib, D, G):
    """Tile n is group n % 2's and lies in stage n % depth.  A group that waits for use k of a stage without having waited for use k - 1 sees
    the same parity as two uses before, so all uses of a stage must be one group's."""
    for cluster in (0, 2, 3, 4, 5, 6, 8, 9, 10, 16):
        for limit in range(48 * 1024, OPTIN + 1, 4096):
            n = lib.pick(D, G, limit, cluster)
            owners = [{t % GROUPS for t in range(s, 4 * GROUPS * n, n)} for s in range(n)]
            assert all(len(o) == 1 for o in owners), (cluster, limit, n)
            if n:
                assert lib.size(D, G, n, cluster) <= limit
                assert n == 8 or lib.size(D, G, n + GROUPS, cluster) > limit        # and no less than fits
        assert lib.pick(D, G, OPTIN, cluster) >= 4                  # on the device itself
