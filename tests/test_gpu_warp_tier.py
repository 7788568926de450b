"""Launches of enough queries for the warp tier (one warp per query): queries
at the edges of its table and of its vector length, ties, saturated counts,
every form it serves.  Each result equals that of the block tiers (the posting
walk forced), which the parity tests pin to the oracle, byte for byte."""
import numpy as np
import pytest

from paper_2510_23679_gb300 import pd, synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    return pd.pd_ctx_create(0)


def both(ctx, call):
    """The call's copied result with the tiers chosen and with them forced."""
    got = call()
    pd.pd_ctx_set_walk(ctx, pd.PD_WALK_MERGE)
    try:
        want = call()
    finally:
        pd.pd_ctx_set_walk(ctx, pd.PD_WALK_AUTO)
    assert len(got) == len(want) and all(np.array_equal(x, y) for x, y in zip(got, want))
    return got


def all_forms(ctx, prof):
    def plain():
        hits = pd.pd_best_hits_all(ctx, prof)
        return (*pd.pd_hits_copy(ctx, hits), pd.pd_bbh_copy(ctx, pd.pd_bbh_all(ctx, prof, hits)))

    rows = both(ctx, plain)
    pd.pd_ctx_set_symmetric(ctx, False)
    try:
        two_sided = both(ctx, plain)
    finally:
        pd.pd_ctx_set_symmetric(ctx, True)
    assert all(np.array_equal(x, y) for x, y in zip(rows, two_sided))
    both(ctx, lambda: pd.pd_hits_copy(ctx, pd.pd_best_hits_shard(ctx, prof, 1, 3)))
    both(ctx, lambda: pd.pd_hits_copy(ctx, pd.pd_paralog_hits(ctx, prof)))
    return rows


def filler(rng, n):
    """n short genes over the whole alphabet."""
    lets = np.frombuffer(synth.ALPHABET, np.uint8)
    return [lets[rng.integers(0, 20, 9)].tobytes() for _ in range(n)]


# occupied slots one below, at and above the most the warp tier lists (832)
@pytest.mark.parametrize("targets", [1, 31, 831, 832, 833, 1500])
def test_listed_slots(ctx, targets):
    rng = np.random.default_rng(targets)
    gene = b"ACDEFGHIKLMNPQRSTVWY"
    # one gene, its copies in another genome (all tied), each with a k-mer of its own
    copies = [gene + filler(rng, 1)[0] for _ in range(targets)]
    ds = synth.from_strings([[gene] + filler(rng, 8000), copies, filler(rng, 9000)])
    prof = pd.pd_build_profiles(ctx, ds.residues, ds.gene_ptr, ds.genome_ptr, 6)
    row_ptr, cols, _, _ = all_forms(ctx, prof)
    assert set(cols[row_ptr[0]:row_ptr[1]].tolist()) <= set(range(8001, 8001 + targets)) and row_ptr[1] >= 1


def test_long_vectors(ctx):
    """Genes of 2040 .. 2060 and 9000 distinct shared k-mers around the most
    entries (2048) a warp takes, and genes whose counts leave no packed slot."""
    rng = np.random.default_rng(5)
    lets = np.frombuffer(synth.ALPHABET, np.uint8)
    long = [lets[rng.integers(0, 20, n + 5)].tobytes() for n in (2040, 2047, 2048, 2049, 2060, 9000)]
    repeats = [b"AC" * 4000, b"AC" * 3999 + b"DE" * 50]
    ds = synth.from_strings([long + repeats + filler(rng, 9000), repeats[::-1] + filler(rng, 8000), long])
    prof = pd.pd_build_profiles(ctx, ds.residues, ds.gene_ptr, ds.genome_ptr, 6)
    row_ptr, cols, s, _ = all_forms(ctx, prof)
    third = int(ds.genome_ptr[2])
    for i, n in enumerate((2040, 2047, 2048, 2049, 2060, 9000)):
        row = {int(c): int(v) for c, v in zip(cols[row_ptr[i]:row_ptr[i + 1]], s[row_ptr[i]:row_ptr[i + 1]])}
        assert row[third + i] == n


@pytest.mark.parametrize("genomes", [2, 511, 512, 513])
def test_genomes(ctx, genomes):
    """Around the most target genomes the warp tier takes, with exact ties
    inside genomes (short genes over two letters)."""
    rng = np.random.default_rng(genomes)
    lets = np.frombuffer(b"ACDE", np.uint8)
    cuts = np.sort(rng.integers(0, 17001, genomes - 1)).tolist()
    genes = [lets[rng.integers(0, 4, 8)].tobytes() for _ in range(17000)]
    ds = synth.from_strings([genes[a:b] for a, b in zip([0] + cuts, cuts + [17000])])
    all_forms(ctx, pd.pd_build_profiles(ctx, ds.residues, ds.gene_ptr, ds.genome_ptr, 7))


def test_saturated_counts(ctx):
    """140000 genes leave 14 bits of count: k-mers repeated more often."""
    rng = np.random.default_rng(9)
    long = [b"A" * 20000 + b"CDEFG", b"A" * 17000 + b"CDEF", b"A" * 16390, b"A" * 100]
    ds = synth.from_strings([long + filler(rng, 70000), [b"C" + g for g in long] + filler(rng, 70000)])
    prof = pd.pd_build_profiles(ctx, ds.residues, ds.gene_ptr, ds.genome_ptr, 5)
    assert pd.pd_profiles_get_info(prof).count_bits == 14
    all_forms(ctx, prof)


def test_split_by_expected_postings(ctx):
    """Lists of more than 8 postings on average: the queries of the first
    genomes and of long genes go to the blocks, the others to the warps."""
    for genomes, genes in ((24, 700), (70, 250)):
        ds = synth.workload("pan50x3000", n_genomes=genomes, genes_per_genome=("fixed", genes), n_families=genes // 2,
                            seed=genomes)
        prof = pd.pd_build_profiles(ctx, ds.residues, ds.gene_ptr, ds.genome_ptr, 5)
        info = pd.pd_profiles_get_info(prof)
        assert info.n_genes >= 16384 and info.n_join >= 8 * info.n_entries
        all_forms(ctx, prof)
