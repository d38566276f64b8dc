"""The room of the tile lists: what the buffers hold, and never more than a saturated offset tells from
a full list. Offsets are ints that saturate at INT_MAX; a tile whose segment [offset, offset + count)
ends beyond the room scans every triangle instead. The function is compiled for the host."""

import os
import subprocess

import pytest

INT_MAX = 2 ** 31 - 1


@pytest.fixture(scope="module")
def room(tmp_path_factory):
    from paper_2104_03989_gb300 import build as B

    d = tmp_path_factory.mktemp("room")
    src, exe = str(d / "room.cu"), str(d / "room")
    with open(src, "w") as f:
        f.write('#include <cstdio>\n#include <cstdlib>\n#include "kernels.cuh"\n'
                "int main(int, char** v) { std::printf(\"%lld\", adms::tile_list_room(std::atoll(v[1]), std::atoll(v[2]))); }\n")
    subprocess.run([B._nvcc()] + B.NVCC_FLAGS + [src, "-o", exe], check=True, env=dict(os.environ))
    return lambda capacity, records: int(subprocess.run([exe, str(capacity), str(records)], check=True,
                                                        capture_output=True, text=True).stdout)


@pytest.mark.parametrize("records", [1, 5000, 1 << 20, 107_374_182, 107_374_183, 200_000_000, 1 << 28, 1 << 29])
@pytest.mark.parametrize("per_triangle", [0, 8, 20])
def test_a_saturated_offset_is_always_beyond_the_room(room, records, per_triangle):
    capacity = per_triangle * records
    got = room(capacity, records)
    assert got == min(capacity + 12 * records, INT_MAX)
    for total in (capacity, got, got + 1, 2 ** 31, 3 * 2 ** 31):  # entries reserved before the tile's own
        offset, count = min(total, INT_MAX), 1
        assert (offset + count > got) == (total + count > got)
