"""The kernels that search for the visible prefixes of a plan: an eighth of the range a step, 8 rows and 4 shards
a warp.  Exact."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gu():
    import gpu_util
    return gpu_util


LENGTHS = [1, 2, 6, 7, 8, 9, 15, 16, 55, 56, 63, 64, 65, 72, 511, 512, 513, 4095, 4096]


@pytest.mark.parametrize("maps,n_q,J", [(1, 15, 2), (1, 16, 1), (3, 33, 4), (2, 200, 40)])
def test_prefixes_of_shards_around_the_powers_of_eight(gu, maps, n_q, J):
    from paper_2507_05228_b200 import binding as cb
    rng = np.random.default_rng(n_q)
    P = len(LENGTHS)
    kv_of = np.stack([rng.permutation(np.repeat(np.arange(P), rng.permutation(LENGTHS))) for _ in range(maps)]).astype(np.int32)
    q_of = rng.integers(0, J, (maps, n_q)).astype(np.int32)  # (some query shards stay empty)
    n_kv = kv_of.shape[1]
    plan = cb.cascade_shard_plan(q_of, kv_of, J, P, q_pos_offset=n_kv - n_q)
    for off in (n_kv - n_q, 0, 300, n_kv - 1, -5):  # the first as the plan was made
        if off != n_kv - n_q:
            plan.advance(off)
        for mp in range(maps):
            ref = oracle.shard_plan(q_of[mp], kv_of[mp], J, P, q_pos_offset=off)
            assert np.array_equal(gu.read_plan_device_array(plan, "vis")[mp], ref.vis), (off, mp)
            assert np.array_equal(gu.read_plan_device_array(plan, "pair_class")[mp], ref.pair_class), (off, mp)
    plan.destroy()
