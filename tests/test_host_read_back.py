"""Where the read-back may write from the host: only memory that CUDA does not know (a
device pointer comes back as an error, managed and pinned memory is copied to as it is),
whatever the other output's memory is.  Sizes: under and over the 4 MiB from which pages
are made by threads, and several chunks."""
import pytest

import host_unit


@pytest.fixture(scope="module")
def prog(tmp_path_factory):
    return host_unit.program(tmp_path_factory, "read_back", "ctd_readback.cpp", "ctd_memory.cpp")


@pytest.mark.parametrize("n", [1 << 20, 2 << 20, (9 << 20) + 24, (33 << 20) + 8])
@pytest.mark.parametrize("kinds", ["nn", "uu", "nu", "un", "mm", "mn", "nm", "dd", "nd", "dn", "ud", "pn", "np", "pm"])
def test_destinations(prog, kinds, n):
    assert host_unit.run(prog, kinds, n) == "ok\n"
