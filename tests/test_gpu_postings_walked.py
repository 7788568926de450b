"""postings_walked counts a query's postings once, whichever tier keeps it: the
automatic tiers report what the block tiers alone do, on every run."""
import numpy as np
import pytest

from paper_2510_23679_gb300 import pd, synth

pytestmark = pytest.mark.gpu

LETTERS = np.frombuffer(synth.ALPHABET, np.uint8)


@pytest.mark.parametrize("copies", [0, 900])
def test_counted_once(copies):
    """With `copies`, the genes of the first genome meet more targets than the
    warp tier's table lists (832): they are walked there and once more."""
    ctx = pd.pd_ctx_create(0)
    rng = np.random.default_rng(copies)
    gene = LETTERS[rng.integers(0, 20, 40)].tobytes()
    filler = [LETTERS[rng.integers(0, 20, 9)].tobytes() for _ in range(18000)]
    ds = synth.from_strings([[gene] * 30 + filler[:9000], [gene + f for f in filler[:copies]] + filler[9000:],
                             filler[:3000]])
    prof = pd.pd_build_profiles(ctx, ds.residues, ds.gene_ptr, ds.genome_ptr, 6)

    def calls():
        jobs = np.array([[0, 1], [0, 2], [1, 2]], np.uint32)
        yield pd.pd_hits_get_info(pd.pd_best_hits_all(ctx, prof))
        yield pd.pd_hits_get_info(pd.pd_best_hits_shard(ctx, prof, 0, 2))
        yield pd.pd_hits_get_info(pd.pd_paralog_hits(ctx, prof))
        yield pd.pd_batch_get_info(pd.pd_bbh_pairs(ctx, prof, jobs))

    got = [[i.postings_walked for i in calls()] for _ in range(3)]
    pd.pd_ctx_set_walk(ctx, pd.PD_WALK_MERGE)
    want = [i.postings_walked for i in calls()]
    assert min(want) > 0 and all(x == want for x in got), (got, want)
