"""Exact ties of the symmetric form: rows with many of them (sorted by a warp up
to 512 entries, by a block in shared memory up to 4096, in place beyond) and
datasets whose number of listed ties changes from run to run by more than a
retry leaves to spare."""
import numpy as np
import pytest

from paper_2510_23679_gb300 import pd, synth

pytestmark = pytest.mark.gpu

LETTERS = np.frombuffer(synth.ALPHABET, np.uint8)


@pytest.fixture(scope="module")
def ctx():
    return pd.pd_ctx_create(0)


def rows(ctx, prof, call):
    hits = call(ctx, prof)
    return (*pd.pd_hits_copy(ctx, hits), pd.pd_bbh_copy(ctx, pd.pd_bbh_all(ctx, prof, hits)))


def equal_to_plain(ctx, prof, call, repeats=1):
    pd.pd_ctx_set_symmetric(ctx, False)
    try:
        want = rows(ctx, prof, call)
    finally:
        pd.pd_ctx_set_symmetric(ctx, True)
    for _ in range(repeats):
        got = rows(ctx, prof, call)
        assert all(np.array_equal(x, y) for x, y in zip(got, want))
    return want


def unfiltered(ctx, prof):
    return pd.pd_best_hits_all(ctx, prof)


def filtered(ctx, prof):
    return pd.pd_best_hits_all_filtered(ctx, prof, (0, 1), (0, 1))


@pytest.mark.parametrize("copies", [2, 509, 510, 511, 512, 1023, 1024, 1025, 4094, 4095, 4097, 9001])
def test_rows_of_many_ties(ctx, copies):
    """Genes with `copies` tied hits in one genome and one or none in two others."""
    rng = np.random.default_rng(copies)
    gene, other = (LETTERS[rng.integers(0, 20, 30)].tobytes() for _ in range(2))
    ds = synth.from_strings([[other], [gene] * copies, [other, gene], [gene, other + b"A", gene + b"C"]])
    prof = pd.pd_build_profiles(ctx, ds.residues, ds.gene_ptr, ds.genome_ptr, 5)
    for call in (unfiltered, filtered):
        row_ptr, cols, _, _ = equal_to_plain(ctx, prof, call)
        last = ds.n_genes - 3  # gene of the last genome: every copy, then the gene of the third genome
        assert cols[row_ptr[last]:row_ptr[last + 1]].tolist() == [*range(1, copies + 1), copies + 2]


def test_number_of_ties_varies(ctx):
    """Random short genes of many genomes: tens of millions of ties with maxima
    that are beaten later, a number that no two runs share."""
    genomes, genes, length = 800, 40, 60
    n = genomes * genes
    residues = LETTERS[np.random.default_rng(1).integers(0, 20, n * length)]
    prof = pd.pd_build_profiles(ctx, residues, np.arange(n + 1, dtype=np.int64) * length,
                                np.arange(genomes + 1, dtype=np.int32) * genes, 3)
    for call in (unfiltered, filtered):
        equal_to_plain(ctx, prof, call, repeats=8)


def test_no_room_for_a_longer_list_of_ties():
    """The plain form, which lists no ties, answers instead."""
    refused = []

    def on_alloc(nbytes):
        if nbytes > 300 << 20:  # the longer list; the maxima take 205 MB, rows 153
            refused.append(nbytes)
        return nbytes <= 300 << 20

    ctx = pd.pd_ctx_create(0, on_alloc=on_alloc)
    genomes, genes, length = 800, 40, 60
    n = genomes * genes
    residues = LETTERS[np.random.default_rng(1).integers(0, 20, n * length)]
    prof = pd.pd_build_profiles(ctx, residues, np.arange(n + 1, dtype=np.int64) * length,
                                np.arange(genomes + 1, dtype=np.int32) * genes, 3)
    equal_to_plain(ctx, prof, unfiltered)
    assert len(refused) == 1


@pytest.mark.parametrize("theta,tau", [((0, 1), (0, 1)), ((3, 4), (0, 1)), ((0, 1), (1, 2)), ((4, 5), (2, 5))])
@pytest.mark.parametrize("genomes,genes", [(2, 1500), (9, 400), (64, 120)])
def test_filtered_of_many_postings(ctx, genomes, genes, theta, tau):
    """Enough postings for the filtered form to walk each pair from one side."""
    rng = np.random.default_rng(genomes)
    lets = np.frombuffer(b"ACD", np.uint8)
    ds = synth.from_strings([[lets[rng.integers(0, 3, int(rng.integers(1, 40)))].tobytes()
                              for _ in range(0 if g == 1 and genomes > 2 else genes)] for g in range(genomes)])
    prof = pd.pd_build_profiles(ctx, ds.residues, ds.gene_ptr, ds.genome_ptr, 3)
    info = pd.pd_profiles_get_info(prof)
    assert info.n_join / 2 >= (8 << 20) + 2 * genomes * ds.n_genes
    want = equal_to_plain(ctx, prof, lambda c, p: pd.pd_best_hits_all_filtered(c, p, theta, tau))
    assert len(want[1])
