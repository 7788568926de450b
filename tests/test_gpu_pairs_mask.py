"""Listed pairs walked genome by genome: target genomes around the words of the
mask, pairs listed twice and both ways round, genomes without genes.  Every
pair's rows and BBH equal the single-pair calls'."""
import numpy as np
import pytest

from paper_2510_23679_gb300 import pd, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("genomes", [2, 31, 32, 33, 65])
def test_masked_targets(genomes):
    ctx = pd.pd_ctx_create(0)
    rng = np.random.default_rng(genomes)
    letters = np.frombuffer(b"ACDEF", np.uint8)
    sizes = rng.integers(0, 12, genomes)
    sizes[[0, genomes - 1]] = 9
    ds = synth.from_strings([[letters[rng.integers(0, 5, 30)].tobytes() for _ in range(n)] for n in sizes])
    prof = pd.pd_build_profiles(ctx, ds.residues, ds.gene_ptr, ds.genome_ptr, 3)
    pairs = rng.integers(0, genomes, (3 * genomes, 2))
    pairs = pairs[pairs[:, 0] != pairs[:, 1]]
    pairs = np.concatenate([pairs, pairs[:4], pairs[:4, ::-1], [[0, genomes - 1]]]).astype(np.uint32)
    batch = pd.pd_bbh_pairs(ctx, prof, pairs)
    row_ptr, cols, s = pd.pd_batch_copy_hits(ctx, batch)
    job_ptr, bbh = pd.pd_batch_copy_bbh(ctx, batch)
    row = 0
    for j, (p, q) in enumerate(pairs.tolist()):
        for x, y in ((p, q), (q, p)):
            rp, c, v = pd.pd_hits_copy(ctx, pd.pd_best_hits(ctx, prof, x, y))
            at = row_ptr[row:row + sizes[x] + 1]
            assert np.array_equal(at - at[0], rp)
            assert np.array_equal(cols[at[0]:at[-1]], c) and np.array_equal(s[at[0]:at[-1]], v)
            row += sizes[x]
        want = pd.pd_bbh_copy(ctx, pd.pd_bbh(ctx, prof, p, q))
        assert np.array_equal(bbh[job_ptr[j]:job_ptr[j + 1]], want)
