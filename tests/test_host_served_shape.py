"""Which served batches share the SMs: small ones among three small ones or more, not a
small one among requests that fill the GPU."""
import pytest

import host_unit

FILL = 1e7


@pytest.fixture(scope="module")
def shares(tmp_path_factory):
    prog = host_unit.program(tmp_path_factory, "served_shape")
    return lambda batch, *running: host_unit.run(prog, FILL, batch, *running) == "1\n"


@pytest.mark.parametrize("batch,running,want", [
    (4e6, (4e6,), False),
    (4e6, (4e6, 4e6), False),
    (4e6, (4e6, 4e6, 4e6), True),
    (4e6, (4e6, 1e3, 9.9e6, 4e6), True),
    (4e6, (4e6, 8e7, 8e7), False),           # alone among large ones
    (4e6, (4e6, 4e6, 8e7), False),
    (4e6, (4e6, 8e7, 4e6, 4e6), True),
    (8e7, (8e7, 4e6, 4e6, 4e6), False),      # a large one never does
    (1e7, (1e7, 4e6, 4e6, 4e6), False),
])
def test_rule(shares, batch, running, want):
    assert shares(batch, *running) is want
