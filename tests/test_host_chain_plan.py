"""How a batched call shares its scratch memory among its requests' chains: streams are
given up only where that makes the tallies fit, whatever the sizes beside a large grid."""
import random

import pytest

import host_unit

BUDGET = 4 << 30   # bytes: 2^29 voxels


@pytest.fixture(scope="module")
def plan(tmp_path_factory):
    prog = host_unit.program(tmp_path_factory, "chain_plan")

    def f(nvox, nb, lanes):
        v = [int(x) for x in host_unit.run(prog, nb, lanes, *nvox).split()]
        return v[0], v[1:1 + len(nvox)], v[1 + len(nvox):]
    return f


@pytest.mark.parametrize("nvox,nb,lanes,want_lanes,want_group", [
    ([256 ** 3] + [24 ** 3] * 63, 10, 64, 64, [10] * 64),           # 1.4 GB in all
    ([256 ** 3] + [64 ** 3] * 24, 20, 25, 25, [16] + [20] * 24),    # 20 batches of 256^3 never fit
    ([512 ** 3] + [24 ** 3] * 63, 10, 64, 64, [2] + [10] * 63),
    ([800 ** 3] + [24 ** 3] * 7, 10, 8, 8, [1] + [10] * 7),         # one tally is over half the budget
    ([256 ** 3] * 64, 10, 64, 3, [10] * 64),                        # three parts of 1.34 GB
    ([256 ** 3] * 6, 20, 6, 2, [16] * 6),
    ([256 ** 3], 30, 1, 1, [30]),
    ([128 ** 3] * 16, 10, 16, 16, [10] * 16),
    ([64 ** 3] * 5, 10, 2, 2, [10] * 5),
])
def test_plans(plan, nvox, nb, lanes, want_lanes, want_group):
    got, group, need = plan(nvox, nb, lanes)
    assert (got, group) == (want_lanes, want_group)
    assert 8 * sum(need) <= BUDGET


def test_random_requests(plan):
    rng = random.Random(3)
    for _ in range(60):
        n, nb = rng.randint(1, 70), rng.choice([2, 3, 10, 40, 300])
        lanes = min(n, rng.choice([1, 2, 5, 64]))
        nvox = [int(2 ** rng.uniform(3, 30)) for _ in range(n)]
        got, group, need = plan(nvox, nb, lanes)
        whole = max(BUDGET // (2 if lanes > 1 else 1) // 8, 1)
        assert 1 <= got <= lanes and len(need) == got and 8 * sum(need) <= BUDGET
        assert group == [max(1, min(nb, whole // v)) for v in nvox]
        parts = [[v * g for k, (v, g) in enumerate(zip(nvox, group)) if k % got == s and g > 1] for s in range(got)]
        assert need == [max(p, default=0) for p in parts]
        if 2 <= got < lanes:   # one stream more would not fit
            more = [max((v * g for k, (v, g) in enumerate(zip(nvox, group)) if k % (got + 1) == s and g > 1), default=0)
                    for s in range(got + 1)]
            assert 8 * sum(more) > BUDGET
