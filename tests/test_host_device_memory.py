"""Device allocations when memory runs out, over a fake device: every allocation of the
library gets what any context of the device holds idle, and nothing that is lent, in use
or on another device; and what a context keeps idle is bounded."""
import pytest

import host_unit


@pytest.fixture(scope="module")
def prog(tmp_path_factory):
    return host_unit.program(tmp_path_factory, "device_memory", "ctd_memory.cpp")


@pytest.mark.parametrize("what", ["c", "n", "o", "kept", "bounded", "threads"])
def test_idle_memory(prog, what):
    assert host_unit.run(prog, what) == "ok\n"
