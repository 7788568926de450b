"""pd_summin_list at the edges of its hash join: vectors around the table's
409 entries and in several parts, runs of pairs of one gene around the 32 that
a warp takes, genes without windows.  Compared with the oracle's definition."""
import numpy as np
import pytest

import oracle
from paper_2510_23679_gb300 import pd, synth

pytestmark = pytest.mark.gpu

# windows of the genes at k = 4, all distinct or nearly so
LENGTHS = [0, 1, 3, 63, 64, 408, 409, 410, 818, 819, 6000]


@pytest.mark.parametrize("pairs", [1, 31, 32, 33, 64, 1000])
def test_pairs(pairs):
    ctx = pd.pd_ctx_create(0)
    rng = np.random.default_rng(pairs)
    lets = np.frombuffer(synth.ALPHABET, np.uint8)
    base = lets[rng.integers(0, 20, max(LENGTHS) + 3)]
    # genes that share a prefix, so that every vector meets the others
    genes = [base[:n + 3].tobytes() if n else b"" for n in LENGTHS]
    other = [g[5:] + b"ACAC" for g in genes]
    ds = synth.from_strings([genes, other])
    prof = pd.pd_build_profiles(ctx, ds.residues, ds.gene_ptr, ds.genome_ptr, 4)
    a = np.sort(rng.integers(0, ds.n_genes, pairs)).astype(np.uint32)
    a[:pairs // 2] = len(LENGTHS) - 1  # a long run of the longest gene
    b = rng.integers(0, ds.n_genes, pairs).astype(np.uint32)
    where = rng.permutation(pairs)
    s, den = pd.pd_summin_list(ctx, prof, a[where], b[where])
    P = oracle.Profiles(ds.residues, ds.gene_ptr, 4)
    want = np.array([P.summin(int(x), int(y)) for x, y in zip(a[where], b[where])])
    assert np.array_equal(s, want[:, 0]) and np.array_equal(den, want[:, 1])
