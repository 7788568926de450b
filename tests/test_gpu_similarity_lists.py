"""pd_summin_list at the edges of its two joins: first vectors around the most
entries a warp takes (818) and around whole parts of both tables (409 and 6553
entries), in either place of the pair, and lists of one pair to several for
every warp.  Also that 32 pairs of long genes are joined side by side and not one
after the other."""
import numpy as np
import pytest

import oracle
from paper_2510_23679_gb300 import pd, synth

pytestmark = pytest.mark.gpu

K = 12


@pytest.fixture(scope="module")
def case():
    """Nucleotide genes of given window counts; every gene has a mutated copy."""
    rng = np.random.default_rng(4)
    letters = np.frombuffer(b"ACGT", np.uint8)
    genes = []
    for n in (1, 408, 409, 410, 817, 818, 819, 4096, 6552, 6553, 6554, 13107, 65535):
        gene = letters[rng.integers(0, 4, n + K - 1)]
        genes.append(gene.tobytes())
        copy = gene.copy()
        at = rng.integers(0, len(gene), max(1, n // 300))
        copy[at] = letters[rng.integers(0, 4, len(at))]
        genes.append(copy.tobytes())
    genes.append((b"ACGTTGCA" * 1200)[:9000])  # few k-mers, many times each
    ds = synth.from_strings([genes, [g for g in genes]])  # every k-mer is shared
    ctx = pd.pd_ctx_create(0)
    return ds, ctx, pd.pd_build_profiles_alphabet(ctx, ds.residues, ds.gene_ptr, ds.genome_ptr, 4, K)


@pytest.fixture(scope="module")
def want(case):
    ds = case[0]
    n = ds.n_genes // 2
    P = oracle.Profiles(ds.residues, ds.gene_ptr, K, 4)
    a, b = np.divmod(np.arange(n * n, dtype=np.uint32), n)
    return a, b, np.array([P.summin(int(x), int(y)) for x, y in zip(a, b)], np.int64)


def check(got, want):
    assert np.array_equal(got[0].astype(np.int64), want[:, 0])
    assert np.array_equal(got[1].astype(np.int64), want[:, 1])


def test_every_pair_of_lengths(case, want):
    _, ctx, prof = case
    a, b, sums = want
    assert (sums[:, 0] > 4000).sum() >= 20
    check(pd.pd_summin_list(ctx, prof, a, b), sums)
    for i in range(0, len(a), 37):  # one pair a call
        check(pd.pd_summin_list(ctx, prof, a[i:i + 1], b[i:i + 1]), sums[i:i + 1])


@pytest.mark.parametrize("pairs", [2, 31, 33, 5471, 5472, 10943, 10945, 200003])
def test_pairs_per_warp(case, want, pairs):
    ds, ctx, prof = case
    a, b, sums = want
    lengths = np.diff(ds.gene_ptr)
    pick = np.flatnonzero(lengths[a] < 5000) if pairs > 6000 else np.arange(len(a))  # keeps the longest list quick
    pick = pick[np.random.default_rng(pairs).integers(0, len(pick), pairs)]
    half = ds.n_genes // 2  # the same genes of the other genome
    check(pd.pd_summin_list(ctx, prof, a[pick] + np.uint32(half) * (pick % 2).astype(np.uint32), b[pick]), sums[pick])


def test_long_pairs_are_not_joined_one_after_the_other(case):
    ds, ctx, prof = case
    long = int(np.argmax(np.diff(ds.gene_ptr)))  # 65535 windows

    def ms(n):
        a, b = np.full(n, long, np.uint32), np.full(n, long + 1, np.uint32)
        best = None
        for _ in range(3):
            pd.pd_ctx_reset_timing(ctx)
            pd.pd_ctx_set_timing(ctx, True)
            pd.pd_summin_list(ctx, prof, a, b)
            pd.pd_ctx_set_timing(ctx, False)
            t = pd.pd_ctx_kernel_time(ctx)[0]
            best = t if best is None else min(best, t)
        return best

    assert ms(32) < 4 * ms(1)  # 32 blocks, far fewer than the chip holds
