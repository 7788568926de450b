"""Device memory of profiles and of a served index: of many windows, and of an
index with a budget, it is the size that the index and the vectors need, not
that of arrays of the dataset's windows."""
import numpy as np
import pytest

from paper_2510_23679_gb300 import pd, synth

pytestmark = pytest.mark.gpu

LETTERS = np.frombuffer(synth.ALPHABET, np.uint8)


def dataset(genomes, genes, length, families, mutated, seed):
    """Genomes of `genes` genes; each a family's sequence with some letters replaced."""
    rng = np.random.default_rng(seed)
    family = LETTERS[rng.integers(0, 20, (families, length))]
    n = genomes * genes
    residues = family[np.concatenate([rng.permutation(families)[:genes] for _ in range(genomes)])]
    other = rng.random(residues.shape, dtype=np.float32) < mutated
    residues[other] = LETTERS[rng.integers(0, 20, int(other.sum()))]
    return (np.ascontiguousarray(residues.reshape(-1)), np.arange(n + 1, dtype=np.int64) * length,
            np.arange(genomes + 1, dtype=np.int32) * genes)


def needed(info, genes, genomes, shared):
    """Bytes of `shared` vector entries, the postings and the k-mers, the genes'
    and genomes' words, and the rounding of each array."""
    return 16 * shared + 4 * info.n_windows + 8 * info.n_distinct + 26 * genes + 4 * genomes + (1 << 14)


# the vectors beside the second buffer of the sort, or after it was given back
@pytest.mark.parametrize("genomes,genes,families,mutated", [(20, 3000, 9000, 0.15), (6, 10000, 10000, 0.0)])
def test_many_windows(genomes, genes, families, mutated):
    ctx = pd.pd_ctx_create(0)
    residues, gene_ptr, genome_ptr = dataset(genomes, genes, 320, families, mutated, 1)
    prof = pd.pd_build_profiles(ctx, residues, gene_ptr, genome_ptr, 6)
    info = pd.pd_profiles_get_info(prof)
    assert info.n_windows > 16 << 20 and info.n_entries <= info.n_windows
    ptr = pd.pd_profiles_copy_index(ctx, prof)[0]
    size = np.diff(ptr)
    shared = int(size[size > 1].sum())
    assert (shared * 4 > info.n_windows * 3) == (mutated == 0.0)
    assert info.device_bytes <= needed(info, genomes * genes, genomes, shared)
    # the vectors hold what the queries need: every copy of a gene is its Best Hit, or
    # the walk that reads them equals the posting lists' own count
    if mutated == 0.0:
        row_ptr, cols, s = pd.pd_hits_copy(ctx, pd.pd_best_hits_all(ctx, prof))
        assert np.array_equal(np.diff(row_ptr), np.full(genomes * genes, genomes - 1))
        assert (s == 320 - 6 + 1).all()
    else:
        pd.pd_ctx_set_symmetric(ctx, False)
        assert pd.pd_hits_get_info(pd.pd_best_hits_all(ctx, prof)).postings_walked == \
            int((size[size > 1].astype(np.int64) ** 2).sum())


@pytest.mark.parametrize("genes,k", [(60, 4), (4000, 6)])
def test_served_index_fits_its_budget(genes, k):
    """A budget of what a dictionary build of the resident genomes took: the
    residues, 18 bytes a window, 4 a k-mer, the dictionary and the genes' words.
    (Vectors take 16 bytes for every k-mer that two genes share, so this holds
    where at most seven eighths are.)"""
    ctx = pd.pd_ctx_create(0)
    genomes = 8
    residues, gene_ptr, genome_ptr = dataset(genomes, genes, 300, 3 * genes, 0.1, 2)
    prof = pd.pd_build_profiles(ctx, residues, gene_ptr, genome_ptr, k)
    info = pd.pd_profiles_get_info(prof)
    size = np.diff(pd.pd_profiles_copy_index(ctx, prof)[0])
    assert size[size > 1].sum() * 8 <= info.n_windows * 7
    dictionary = -(-20 ** k // 224) * 32
    budget = max(len(residues), 1 << 20) + 18 * info.n_windows + 4 * info.n_distinct + dictionary + \
        26 * genes * genomes + (1 << 14)
    index = pd.pd_index_create(ctx, residues, gene_ptr, genome_ptr, k, budget)
    assert pd.pd_index_get_info(index).device_bytes <= budget
    index.free()
