"""Profiles built by sorting, at the edges of the sort's tiles: window totals
around a tile, posting lists and repeated k-mers that run across tiles, counts
that do not fit a posting, many tiny and empty genomes, genes whose ids leave
no room for the code in a sort record.  The index and the vectors are compared
with numpy's sort of all (code, gene) windows, entry by entry; sum-min and the
Best Hits with the oracle."""
import numpy as np
import pytest

import oracle
from paper_2510_23679_gb300 import pd, synth
from tests._gpu import DeviceRun, csr_lists, oracle_nonzero

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    return pd.pd_ctx_create(0)


def windows_of(ds, k, letters=synth.ALPHABET):
    """(codes, genes) of every window, in gene order."""
    number = np.zeros(256, np.int64)
    number[list(letters)] = np.arange(len(letters))
    codes, genes = [], []
    for g in range(ds.n_genes):
        d = number[ds.residues[ds.gene_ptr[g]:ds.gene_ptr[g + 1]]]
        if len(d) < k:
            continue
        c = np.zeros(len(d) - k + 1, np.int64)
        for t in range(k):
            c = c * len(letters) + d[t:len(d) - k + 1 + t]
        codes.append(c)
        genes.append(np.full(len(c), g))
    return (np.concatenate(codes), np.concatenate(genes)) if codes else (np.zeros(0, np.int64), np.zeros(0, np.int64))


def check_profiles(ctx, ds, k, prof):
    codes, genes = windows_of(ds, k)
    key, count = np.unique(codes * ds.n_genes + genes, return_counts=True)
    code, gene = key // ds.n_genes, key % ds.n_genes
    distinct, first, size = np.unique(code, return_index=True, return_counts=True)
    info = pd.pd_profiles_get_info(prof)
    assert (info.n_windows, info.n_entries, info.n_distinct) == (len(codes), len(key), len(distinct))
    assert info.max_posting == (size.max() if len(size) else 0)
    assert info.n_join == int((size.astype(np.int64) ** 2).sum())
    ptr, c, g, n = pd.pd_profiles_copy_index(ctx, prof)
    assert np.array_equal(c, distinct) and np.array_equal(ptr, np.append(first, len(key)))
    assert np.array_equal(g, gene) and np.array_equal(n, count)
    by_gene = np.lexsort((code, gene))
    ptr, c, n, La = pd.pd_profiles_copy_mv(ctx, prof)
    assert np.array_equal(c, code[by_gene]) and np.array_equal(n, count[by_gene])
    assert np.array_equal(ptr, np.append(0, np.cumsum(np.bincount(gene, minlength=ds.n_genes))))
    assert np.array_equal(La, np.bincount(genes, minlength=ds.n_genes))


def dataset(rng, lengths, letters, genomes):
    """Genes of the given lengths over a few letters, cut into genomes."""
    lets = np.frombuffer(letters, np.uint8)
    genes = [lets[rng.integers(0, len(lets), n)].tobytes() for n in lengths]
    cuts = np.sort(rng.integers(0, len(genes) + 1, genomes - 1)).tolist()
    return synth.from_strings([genes[a:b] for a, b in zip([0] + cuts, cuts + [len(genes)])])


# window totals one below, at and one above the tiles of the sort (7680), of
# the pass over the sorted records (8192) and its halves, and several of each
@pytest.mark.parametrize("total", [1, 31, 4095, 4096, 4097, 7679, 7680, 7681, 8191, 8192, 8193, 15360, 15361, 40961])
@pytest.mark.parametrize("letters,k", [(b"AC", 1), (b"ACD", 3), (synth.ALPHABET, 2), (synth.ALPHABET, 8)])
def test_window_totals(ctx, total, letters, k):
    rng = np.random.default_rng(total * 100 + k)
    lengths, left = [], total
    while left:
        n = min(left, int(rng.integers(1, 900)))
        lengths += [n + k - 1] + [int(x) for x in rng.integers(0, k, rng.integers(0, 3))]  # and genes of no window
        left -= n
    ds = dataset(rng, lengths, letters, 3)
    run = DeviceRun(ctx, ds, k, device_inputs=total % 2 == 0)
    check_profiles(ctx, ds, k, run.prof)


@pytest.mark.parametrize("k", [1, 4])
def test_repeats_across_tiles(ctx, k):
    """The longest genes allowed, of one letter (a k-mer 65535 times), beside
    genes that share it a few times: runs over many tiles, saturated counts in
    one dataset with 28 and one with 14 count bits."""
    long = b"A" * (65535 + k - 1)
    genes = [[long, b"ACDA" * 5, b"A" * k], [b"C" * 30, long[:30000], b"A" * (k + 3)], [], [b"AAC" * 9, long]]
    ds = synth.from_strings(genes)
    check_profiles(ctx, ds, k, DeviceRun(ctx, ds, k).prof)
    ds = synth.from_strings(genes + [[b"D" * 9] * 140000])
    run = DeviceRun(ctx, ds, k)
    assert run.info.count_bits == 14
    check_profiles(ctx, ds, k, run.prof)
    for gi, gj in ((0, 1), (0, 3), (3, 1)):
        R = oracle.pair_for_dataset(ds, gi, gj, k)
        assert run.summin(gi, gj) == oracle_nonzero(R)
        assert run.best_hits(gi, gj)[0] == csr_lists(R.row_ptr, R.row_col)


@pytest.mark.parametrize("genomes", [4096, 700])
def test_tiny_genomes(ctx, genomes):
    """Up to 4096 genomes of no, one and several genes over short lists of
    letters: lists with many genomes, runs of one genome, and of genomes that
    hold no gene at all."""
    rng = np.random.default_rng(genomes)
    ds = dataset(rng, rng.integers(0, 40, 5000), b"ACDE", genomes)
    run = DeviceRun(ctx, ds, 2)
    check_profiles(ctx, ds, 2, run.prof)
    sizes = ds.genome_sizes()
    big = np.argsort(sizes)[-3:]
    for gi, gj in ((int(big[0]), int(big[1])), (int(big[2]), int(big[0]))):
        R = oracle.pair_for_dataset(ds, gi, gj, 2)
        assert run.best_hits(gi, gj)[0] == csr_lists(R.row_ptr, R.row_col)
    hits = pd.pd_best_hits_all(ctx, run.prof)
    pd.pd_ctx_set_symmetric(ctx, False)
    try:
        plain = pd.pd_best_hits_all(ctx, run.prof)
    finally:
        pd.pd_ctx_set_symmetric(ctx, True)
    for x, y in zip(pd.pd_hits_copy(ctx, hits), pd.pd_hits_copy(ctx, plain)):
        assert np.array_equal(x, y)


def test_gene_beside_itself(ctx):
    """Sum-min of a gene with itself counts the k-mers that only it has."""
    ds = synth.from_strings([[b"ACDEFGHIKL", b"AC"], [b"ACDEFMNPQR"]])
    run = DeviceRun(ctx, ds, 3)
    s, den = pd.pd_summin_list(ctx, run.prof, np.array([0, 0, 1, 2], np.uint32), np.array([0, 2, 1, 2], np.uint32))
    assert s.tolist() == [8, 3, 0, 8] and den.tolist() == [8, 13, 0, 8]


def test_more_genes_than_a_record_holds(ctx):
    """2^29 genes, nearly all empty, at k = 8: 35 bits of code and 30 of gene
    are sorted in two slices.  The result is that of the genes alone."""
    import torch
    small = synth.workload("pan4x250", n_genomes=2, genes_per_genome=("fixed", 60), n_families=50, seed=21)
    empty, cut = 1 << 29, int(small.genome_ptr[1])
    gp = torch.from_numpy(small.gene_ptr).cuda()
    gene_ptr = torch.cat([gp[:cut + 1], gp[cut].expand(empty), gp[cut + 1:]])
    shift = np.where(np.arange(small.n_genes) < cut, 0, empty)
    genome_ptr = np.array([0, cut, cut + empty, empty + small.n_genes], np.int32)
    prof = pd.pd_build_profiles(ctx, torch.from_numpy(small.residues).cuda(), gene_ptr, genome_ptr, 8)
    ref = DeviceRun(ctx, small, 8)
    got, want = pd.pd_profiles_copy_index(ctx, prof), pd.pd_profiles_copy_index(ctx, ref.prof)
    assert np.array_equal(got[0], want[0]) and np.array_equal(got[1], want[1])
    assert np.array_equal(got[2], want[2] + shift[want[2]]) and np.array_equal(got[3], want[3])
    for x, y in zip(pd.pd_hits_copy(ctx, pd.pd_best_hits(ctx, prof, 0, 2)),
                    pd.pd_hits_copy(ctx, pd.pd_best_hits(ctx, ref.prof, 0, 1))):
        assert np.array_equal(x, y)
