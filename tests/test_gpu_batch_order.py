"""Batched jobs, whose posting lists stand in order of k-mer and then job: at
every k, for one job, a power of two of them and one more, rows and BBH pairs
equal those of the same pairs of one profiled dataset."""
import numpy as np
import pytest

from paper_2510_23679_gb300 import pd, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("jobs", [1, 2, 16, 17, 64])
@pytest.mark.parametrize("k", [1, 2, 3, 4, 5, 6, 7, 8])
def test_jobs(k, jobs):
    ctx = pd.pd_ctx_create(0)
    rng = np.random.default_rng(k * 100 + jobs)
    lets = np.frombuffer(synth.ALPHABET, np.uint8)
    core = [lets[rng.integers(0, 20, 60)].tobytes() for _ in range(30)]  # families, a third of them cut short
    genomes = [[core[x][:int(rng.integers(1, 61))] if rng.integers(3) == 0 else core[x]
                for x in rng.integers(0, 30, int(rng.integers(0, 50)))] for _ in range(9)]
    genomes.append([b"A" * 70, b"A" * 900, b"W" * 40 + b"A" * 12])
    ds = synth.from_strings(genomes)
    pairs = rng.integers(0, 10, (4 * jobs, 2))
    pairs = np.concatenate([[[9, 0]], pairs[pairs[:, 0] != pairs[:, 1]]])[:jobs].astype(np.uint32)
    got = pd.pd_bbh_batch(ctx, ds.residues, ds.gene_ptr, ds.genome_ptr, pairs, np.full(len(pairs), k, np.int32))
    prof = pd.pd_build_profiles(ctx, ds.residues, ds.gene_ptr, ds.genome_ptr, k)
    want = pd.pd_bbh_pairs(ctx, prof, pairs)
    for x, y in zip([*pd.pd_batch_copy_hits(ctx, got), *pd.pd_batch_copy_bbh(ctx, got)],
                    [*pd.pd_batch_copy_hits(ctx, want), *pd.pd_batch_copy_bbh(ctx, want)]):
        assert np.array_equal(x, y)
