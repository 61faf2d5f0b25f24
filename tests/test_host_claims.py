"""The claims of a launch's warps and the pieces of a launch that crosses 2^32 histories:
they cover the range once, start in the right batch and tally, and claim by the rule (a
sixteenth of a warp's share raised to a multiple of 32, at most the chunk, when the launch
is alone, else the chunk; 32 for the last 256 per warp), each piece by its own size."""
import pytest

import host_unit

HI = 1 << 32


@pytest.fixture(scope="module")
def launches(tmp_path_factory):
    prog = host_unit.program(tmp_path_factory, "claims", "ctd_claims.cpp", "ctd_memory.cpp")

    def f(*args):
        keys = ("h0", "h1", "b0", "tally", "big", "small", "h_big", "h_hi", "cleared")
        return [dict(zip(keys, map(int, line.split()))) for line in host_unit.run(prog, *args).splitlines()]
    return f


@pytest.mark.parametrize("alone", [0, 1])
@pytest.mark.parametrize("n,nb,h0,h1,chunk,warps", [
    (100_000, 10, 0, 100_000, 256, 5472),
    (2_801_663, 3, 0, 2_801_663, 256, 5472),      # 32 and 64 meet at 2801664
    (2_801_664, 3, 0, 2_801_664, 256, 5472),
    (50_000_000, 7, 0, 50_000_000, 256, 5472),
    (1_500_001, 4, 7, 1_500_001, 40, 5472),
    (1_500_001, 4, 0, 1_500_001, 20, 5472),
    (4 * HI + 5, 7, HI - 3_000_000, HI + 5_000_000, 256, 5472),
    (4 * HI + 5, 7, 3 * HI - 1, 3 * HI + 1, 256, 5472),
    (4 * HI + 5, 3, 0, 4 * HI + 5, 256, 5472),
    (10 * HI, 1000, HI + 17, 3 * HI, 256, 64),
])
def test_pieces_and_claims(launches, n, nb, h0, h1, chunk, warps, alone):
    n_lo, rem = divmod(n, nb)
    start = lambda b: b * n_lo + min(b, rem)
    out = launches(n, nb, h0, h1, chunk, warps, alone)
    assert out[0]["h0"] == h0 and out[-1]["h1"] == h1
    assert all(a["h1"] == b["h0"] and b["h0"] % HI == 0 for a, b in zip(out, out[1:]))
    for k, l in enumerate(out):
        size = l["h1"] - l["h0"]
        assert l["h0"] >> 32 == (l["h1"] - 1) >> 32 == l["h_hi"] and l["cleared"] == k
        assert start(l["b0"]) <= l["h0"] < start(l["b0"] + 1)
        assert l["tally"] == 1000 * (l["b0"] - out[0]["b0"])
        share = size // (16 * warps)
        assert l["big"] == (min((share // 32 + 1) * 32, chunk) if alone else chunk)
        assert l["small"] == min(32, chunk)
        assert l["h_big"] == max(l["h1"] - 256 * warps, l["h0"])
