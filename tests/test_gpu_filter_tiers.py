"""Filtered Best Hits at the edges of the filtered tiers' tables: as many
targets as the packed table lists (2560), one more, more than the split table
holds.  A filter that every candidate passes gives the unfiltered result; one
that cuts by shared occurrences and by length gives the definition's."""
from fractions import Fraction

import numpy as np
import pytest

import oracle
from paper_2510_23679_gb300 import pd, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("targets", [1, 2559, 2560, 2561, 4096, 5000])
def test_targets(targets):
    ctx = pd.pd_ctx_create(0)
    rng = np.random.default_rng(targets)
    lets = np.frombuffer(synth.ALPHABET, np.uint8)
    core = b"ACDEFGHIKL"
    # targets share the query's core and differ in length and repeats
    copies = [core + lets[rng.integers(0, 20, int(rng.integers(0, 9)))].tobytes() for _ in range(targets)]
    ds = synth.from_strings([[core + b"MNPQRS", core * 3], copies])
    k = 3
    prof = pd.pd_build_profiles(ctx, ds.residues, ds.gene_ptr, ds.genome_ptr, k)
    plain = pd.pd_hits_copy(ctx, pd.pd_best_hits(ctx, prof, 0, 1))
    for x, y in zip(plain, pd.pd_hits_copy(ctx, pd.pd_best_hits_filtered(ctx, prof, 0, 1, (1, 1000), (1, 100000)))):
        assert np.array_equal(x, y)
    theta, tau = (3, 4), (1, 2)
    got = pd.pd_hits_copy(ctx, pd.pd_best_hits_filtered(ctx, prof, 0, 1, theta, tau))
    P = oracle.Profiles(ds.residues, ds.gene_ptr, k)
    mv = [dict(zip(*(lambda m, c: (m, c.tolist()))(*P.mv(g)))) for g in range(ds.n_genes)]
    length = np.diff(ds.gene_ptr)
    for a in range(2):
        best, row = Fraction(0), []
        for b in range(targets):
            x, y = mv[a], mv[2 + b]
            shared = x.keys() & y.keys()
            s = sum(min(x[w], y[w]) for w in shared)
            la, lb = int(length[a]), int(length[2 + b])
            if s == 0 or la * theta[1] < theta[0] * lb or lb * theta[1] < theta[0] * la:
                continue
            if sum(x[w] for w in shared) * tau[1] < tau[0] * P.La(a) or \
                    sum(y[w] for w in shared) * tau[1] < tau[0] * P.La(2 + b):
                continue
            r = Fraction(s, P.La(a) + P.La(2 + b) - s)
            if r > best:
                best, row = r, []
            if r == best:
                row.append((b, s))
        assert list(zip(got[1][got[0][a]:got[0][a + 1]].tolist(), got[2][got[0][a]:got[0][a + 1]].tolist())) == row


def test_counts_that_do_not_fit_a_posting():
    """The directional sums hold the target's own multiplicity, also where it
    does not fit a posting (14 bits among 140 000 genes): A x 10000 against A x
    65535, all of whose windows are shared, passes tau = 9/10 both ways."""
    ctx = pd.pd_ctx_create(0)
    ds = synth.from_strings([[b"A" * 10000, b"A" * 65535], [b"A" * 65535, b"A" * 9000 + b"C" * 30000],
                             [b"D" * 9] * 140000])
    prof = pd.pd_build_profiles(ctx, ds.residues, ds.gene_ptr, ds.genome_ptr, 1)
    assert pd.pd_profiles_get_info(prof).count_bits == 14
    ptr, col, s = pd.pd_hits_copy(ctx, pd.pd_best_hits_filtered(ctx, prof, 0, 1, (0, 1), (9, 10)))
    assert (ptr.tolist(), col.tolist(), s.tolist()) == ([0, 1, 2], [0, 0], [10000, 65535])
    ptr, col, s = pd.pd_hits_copy(ctx, pd.pd_best_hits_filtered(ctx, prof, 0, 1, (0, 1), (1, 5)))
    assert (ptr.tolist(), col.tolist(), s.tolist()) == ([0, 1, 2], [1, 0], [9000, 65535])


@pytest.mark.parametrize("theta,tau", [((0, 1), (0, 1)), ((3, 4), (0, 1)), ((0, 1), (1, 2)), ((4, 5), (2, 5))])
@pytest.mark.parametrize("genomes,letters,k", [(2, b"AC", 3), (9, b"ACD", 3), (64, synth.ALPHABET, 2)])
def test_walked_from_one_side(genomes, letters, k, theta, tau):
    """All pairs walked from one side give the rows and BBH pairs of the form
    that walks both, on data full of exact ties and with genomes without genes."""
    ctx = pd.pd_ctx_create(0)
    rng = np.random.default_rng(genomes)
    lets = np.frombuffer(letters, np.uint8)
    genes = [[lets[rng.integers(0, len(lets), int(rng.integers(1, 40)))].tobytes()
              for _ in range(0 if g == 1 and genomes > 2 else int(rng.integers(20, 90)))] for g in range(genomes)]
    ds = synth.from_strings(genes)
    prof = pd.pd_build_profiles(ctx, ds.residues, ds.gene_ptr, ds.genome_ptr, k)
    out = []
    for symmetric in (True, False):
        pd.pd_ctx_set_symmetric(ctx, symmetric)
        hits = pd.pd_best_hits_all_filtered(ctx, prof, theta, tau)
        out.append([*pd.pd_hits_copy(ctx, hits), pd.pd_bbh_copy(ctx, pd.pd_bbh_all(ctx, prof, hits))])
    for x, y in zip(*out):
        assert np.array_equal(x, y)
    assert len(out[0][1])
