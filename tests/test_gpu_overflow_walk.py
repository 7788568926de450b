"""Queries that meet far more targets than a tier's table holds: their walk ends
where the table is full, and queries expected to overflow the warp tier are not
walked there first.  Results equal those of the other forms; the times are
compared with those of launches of the same run."""
import numpy as np
import pytest

from paper_2510_23679_gb300 import pd, synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    return pd.pd_ctx_create(0)


def dataset(genomes, genes, length, seed):
    """Unrelated genes: at small k each meets nearly every other."""
    n = genomes * genes
    letters = np.frombuffer(synth.ALPHABET, np.uint8)
    return (letters[np.random.default_rng(seed).integers(0, 20, n * length)], np.arange(n + 1, dtype=np.int64) * length,
            np.arange(genomes + 1, dtype=np.int32) * genes)


def kernel_ms(ctx, call, *names):
    """Least of three: device ms of the named kernels (all without a name)."""
    call()
    best = None
    for _ in range(3):
        pd.pd_ctx_reset_timing(ctx)
        pd.pd_ctx_set_timing(ctx, True)
        call()
        pd.pd_ctx_set_timing(ctx, False)
        ms = [pd.pd_ctx_kernel_time(ctx, name)[0] for name in names or (None,)]
        best = ms if best is None else [min(x, y) for x, y in zip(best, ms)]
    return best


def forced(ctx, walk, call):
    pd.pd_ctx_set_walk(ctx, walk)
    try:
        return call()
    finally:
        pd.pd_ctx_set_walk(ctx, pd.PD_WALK_AUTO)


def test_full_tables_end_the_walk(ctx):
    prof = pd.pd_build_profiles(ctx, *dataset(10, 2000, 340, 1), 4)
    results = []
    for symmetric in (True, False):
        pd.pd_ctx_set_symmetric(ctx, symmetric)
        for walk in (pd.PD_WALK_AUTO, pd.PD_WALK_MERGE, pd.PD_WALK_WARP):
            results.append(forced(ctx, walk, lambda: pd.pd_hits_copy(ctx, pd.pd_best_hits_all(ctx, prof))))
            # tier 2 takes nearly every query too, and four times as many targets
            t1, t2 = forced(ctx, walk, lambda: kernel_ms(ctx, lambda: pd.pd_best_hits_all(ctx, prof), "summin_bh",
                                                         "summin_bh_t2"))
            assert t1 < 2 * t2, (symmetric, walk, t1, t2)
    pd.pd_ctx_set_symmetric(ctx, True)
    for got in results[1:]:
        assert all(np.array_equal(x, y) for x, y in zip(got, results[0]))


def test_heavy_queries_pass_by_the_warp_tier(ctx):
    """Paralogs, listed pairs and batched jobs of many postings a query take no
    longer than with the block tiers alone."""
    data = dataset(4, 6000, 300, 2)
    prof = pd.pd_build_profiles(ctx, *data, 4)
    pairs = np.array([[0, 1], [2, 3]], np.uint32)
    calls = (lambda: pd.pd_hits_copy(ctx, pd.pd_paralog_hits(ctx, prof)),
             lambda: pd.pd_batch_copy_hits(ctx, pd.pd_bbh_pairs(ctx, prof, pairs)),
             lambda: pd.pd_batch_copy_hits(ctx, pd.pd_bbh_batch(ctx, *data, pairs, np.array([4, 4], np.int32))))
    for call in calls:
        got, want = call(), forced(ctx, pd.PD_WALK_MERGE, call)
        assert all(np.array_equal(x, y) for x, y in zip(got, want))
        ours, = kernel_ms(ctx, call)
        blocks, = forced(ctx, pd.PD_WALK_MERGE, lambda: kernel_ms(ctx, call))
        assert ours < 1.2 * blocks, (ours, blocks)
