"""The warp tier with two lanes a list, outside the symmetric form: an index far
larger than L2 (at least 512 MB of postings) with lists of more than 16 postings
on average.  Rows equal those of the block tiers."""
import numpy as np
import pytest

from paper_2510_23679_gb300 import pd, synth

pytestmark = pytest.mark.gpu


def test_long_lists_of_a_large_index():
    genomes, genes, length, families = 40, 12000, 300, 9000
    rng = np.random.default_rng(7)
    letters = np.frombuffer(synth.ALPHABET, np.uint8)
    family = letters[rng.integers(0, 20, (families, length))]
    n = genomes * genes
    residues = family[rng.integers(0, families, n)]
    at = rng.integers(0, residues.size, residues.size // 50)  # 2% of the letters replaced
    residues.reshape(-1)[at] = letters[rng.integers(0, 20, len(at))]
    ctx = pd.pd_ctx_create(0)
    prof = pd.pd_build_profiles(ctx, residues.reshape(-1), np.arange(n + 1, dtype=np.int64) * length,
                                np.arange(genomes + 1, dtype=np.int32) * genes, 6)
    info = pd.pd_profiles_get_info(prof)
    assert info.n_entries * 4 >= 512 << 20 and info.n_join >= 16 * info.n_entries
    pairs = np.array([[0, 1], [39, 2], [5, 17]], np.uint32)

    def calls():
        yield pd.pd_hits_copy(ctx, pd.pd_best_hits_shard(ctx, prof, 1, 16))
        yield pd.pd_hits_copy(ctx, pd.pd_paralog_hits(ctx, prof))
        yield pd.pd_batch_copy_hits(ctx, pd.pd_bbh_pairs(ctx, prof, pairs))

    pd.pd_ctx_reset_timing(ctx)
    pd.pd_ctx_set_timing(ctx, True)
    got = list(calls())
    pd.pd_ctx_set_timing(ctx, False)
    assert pd.pd_ctx_kernel_time(ctx, "summin_warp")[1] == 3
    pd.pd_ctx_set_walk(ctx, pd.PD_WALK_MERGE)
    for x, y in zip(got, calls()):
        assert len(x[1]) and all(np.array_equal(a, b) for a, b in zip(x, y))
