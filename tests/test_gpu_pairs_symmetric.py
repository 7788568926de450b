"""Listed pairs and batched jobs walked from one side: rows, sums and BBH pairs
equal those of the form that walks both (whole numbers, so exactly), on
datasets full of exact ties, with jobs in either order, listed twice and of
genomes without genes; one job of each against the oracle."""
import numpy as np
import pytest

import oracle
from paper_2510_23679_gb300 import pd, synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    return pd.pd_ctx_create(0)


def dataset(rng, sizes, letters, longest):
    lets = np.frombuffer(letters, np.uint8)
    return synth.from_strings([[lets[rng.integers(0, len(lets), int(rng.integers(1, longest)))].tobytes()
                                for _ in range(n)] for n in sizes])


def both(ctx, call):
    def result(symmetric):
        pd.pd_ctx_set_symmetric(ctx, symmetric)
        try:
            b = call()
        finally:
            pd.pd_ctx_set_symmetric(ctx, True)
        info = pd.pd_batch_get_info(b)
        return [*pd.pd_batch_copy_hits(b.ctx, b), *pd.pd_batch_copy_bbh(b.ctx, b)], info
    (one, one_info), (two, two_info) = result(True), result(False)
    for x, y in zip(one, two):
        assert np.array_equal(x, y)
    assert (one_info.n_hits, one_info.n_bbh) == (two_info.n_hits, two_info.n_bbh)
    assert one_info.postings_walked < 0.7 * two_info.postings_walked  # the other route was taken
    return one


def check_oracle(ds, result, job, k, row0, at):
    ptr, cols, s, job_ptr, pairs = result
    R = oracle.pair_for_dataset(ds, int(job[0]), int(job[1]), k)
    for a in range(R.S.shape[0]):
        assert cols[ptr[row0 + a]:ptr[row0 + a + 1]].tolist() == R.row_bh(a).tolist()
    assert pairs[job_ptr[at]:job_ptr[at + 1]].tolist() == np.asarray(R.bbh).tolist()


@pytest.mark.parametrize("genomes,genes,letters,k,jobs", [
    (33, 70, b"AC", 3, 200),   # two words of partners, every gene shares k-mers with every other
    (64, 40, b"ACD", 4, 900),
    (40, 120, b"ACDEFGHIKLMNPQRSTVWY", 2, 300),
])
def test_listed_pairs(ctx, genomes, genes, letters, k, jobs):
    rng = np.random.default_rng(genomes)
    sizes = rng.integers(genes // 2, genes * 2, genomes)
    sizes[[0, 7, genomes - 1]] = 0, 1, genes
    ds = dataset(rng, sizes, letters, 60)
    prof = pd.pd_build_profiles(ctx, ds.residues, ds.gene_ptr, ds.genome_ptr, k)
    pairs = rng.integers(0, genomes, (jobs, 2))
    pairs = pairs[pairs[:, 0] != pairs[:, 1]]
    pairs = np.concatenate([pairs, pairs[:3], pairs[3:5, ::-1], [[0, 5], [genomes - 1, 0]]]).astype(np.uint32)
    got = both(ctx, lambda: pd.pd_bbh_pairs(ctx, prof, pairs))
    sizes = np.diff(ds.genome_ptr)
    rows = np.concatenate([[0], np.cumsum(sizes[pairs].sum(1))])
    check_oracle(ds, got, pairs[1], k, int(rows[1]), 1)


def test_last_genome_against_all(ctx):
    """Every pair names the last genome (it is never a query), then the first (the only one)."""
    rng = np.random.default_rng(5)
    ds = dataset(rng, [200] * 40, synth.ALPHABET, 27)
    prof = pd.pd_build_profiles(ctx, ds.residues, ds.gene_ptr, ds.genome_ptr, 2)
    for hub in (39, 0):
        pairs = np.array([[hub, g] if g % 2 else [g, hub] for g in range(40) if g != hub], np.uint32)
        got = both(ctx, lambda: pd.pd_bbh_pairs(ctx, prof, pairs))
        check_oracle(ds, got, pairs[3], 2, 3 * 400, 3)


@pytest.mark.parametrize("query_order", [0, 1])
def test_batched_jobs(ctx, query_order):
    rng = np.random.default_rng(9)
    ds = dataset(rng, [400, 380, 0, 1, 500, 420, 390, 410], b"ACD", 70)
    jobs = np.array([[0, 1], [4, 5], [5, 4], [6, 7], [2, 0], [3, 1], [0, 6], [7, 1]], np.uint32)
    ks = np.array([3, 4, 3, 4, 3, 4, 3, 4], np.int32)
    got = both(ctx, lambda: pd.pd_bbh_batch(ctx, ds.residues, ds.gene_ptr, ds.genome_ptr, jobs, ks,
                                            query_order=query_order))
    check_oracle(ds, got, jobs[0], 3, 0, 0)


class Refuse:
    def __init__(self):
        self.calls = self.at = 0

    def on_alloc(self, nbytes):
        self.calls += 1
        return self.calls != self.at


@pytest.mark.parametrize("form", ["pairs", "batch", "filtered"])
def test_no_room_for_the_maxima(form):
    """Each allocation of a call refused in turn: the call reports it, or finds
    room for the form that walks both sides and gives the same result."""
    refuse = Refuse()
    ctx = pd.pd_ctx_create(0, on_alloc=refuse.on_alloc)
    rng = np.random.default_rng(3)
    ds = dataset(rng, [150] * 12 + [0], b"ACD", 50)
    if form == "batch":
        ds = dataset(rng, [900, 900, 0], b"ACD", 60)
    prof = pd.pd_build_profiles(ctx, ds.residues, ds.gene_ptr, ds.genome_ptr, 3)
    pairs = np.array([(a, b) for a in range(12) for b in range(a)], np.uint32)

    def call():
        if form == "filtered":
            hits = pd.pd_best_hits_all_filtered(ctx, prof, (1, 2), (1, 4))
            return [*pd.pd_hits_copy(ctx, hits), pd.pd_bbh_copy(ctx, pd.pd_bbh_all(ctx, prof, hits))]
        if form == "pairs":
            b = pd.pd_bbh_pairs(ctx, prof, pairs)
        else:
            b = pd.pd_bbh_batch(ctx, ds.residues, ds.gene_ptr, ds.genome_ptr, np.array([[0, 1]], np.uint32),
                                np.array([3], np.int32))
        return [*pd.pd_batch_copy_hits(ctx, b), *pd.pd_batch_copy_bbh(ctx, b)]

    refuse.calls = 0
    want, total, found_room = call(), refuse.calls, 0
    for at in range(1, total + 1):
        refuse.calls, refuse.at = 0, at
        try:
            got = call()
        except pd.PdError as err:
            assert err.status == 5
            continue
        found_room += 1
        assert all(np.array_equal(x, y) for x, y in zip(got, want))
    assert found_room
    refuse.at = 0
    assert all(np.array_equal(x, y) for x, y in zip(call(), want))
