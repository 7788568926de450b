"""pd_profiles_copy_mv where a few k-mers are in nearly every gene: posting lists
that cover many of the export's tiles (2048 postings), and ends of lists and of
the index at the edges of a tile."""
import numpy as np
import pytest

from paper_2510_23679_gb300 import pd, synth
from tests.test_gpu_index_sort import check_profiles

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    return pd.pd_ctx_create(0)


@pytest.mark.parametrize("genes", [2047, 2048, 2049, 4096, 30001])
@pytest.mark.parametrize("letters,k", [(b"A", 1), (b"AC", 1), (b"ACD", 2)])
def test_long_lists(ctx, genes, letters, k):
    rng = np.random.default_rng(genes)
    lets = np.frombuffer(letters, np.uint8)
    ds = synth.from_strings([[lets[rng.integers(0, len(lets), 12)].tobytes() for _ in range(genes)], [letters * 400]])
    check_profiles(ctx, ds, k, pd.pd_build_profiles(ctx, ds.residues, ds.gene_ptr, ds.genome_ptr, k))


def test_long_lists_are_shared_out(ctx):
    """Twenty lists of 100000 genes take no more than the sort of the vectors by
    a wide margin, where one thread a list took hundreds of times as long."""
    n, length = 100000, 100
    letters = np.frombuffer(synth.ALPHABET, np.uint8)
    prof = pd.pd_build_profiles(ctx, letters[np.random.default_rng(1).integers(0, 20, n * length)],
                                np.arange(n + 1, dtype=np.int64) * length, np.array([0, n // 2, n], np.int32), 1)
    pd.pd_profiles_copy_mv(ctx, prof)
    pd.pd_ctx_reset_timing(ctx)
    pd.pd_ctx_set_timing(ctx, True)
    pd.pd_profiles_copy_mv(ctx, prof)
    pd.pd_ctx_set_timing(ctx, False)
    keys, sort = (pd.pd_ctx_kernel_time(ctx, name)[0] for name in ("export_mv_keys", "export_mv_sort"))
    assert keys < 10 * sort, (keys, sort)
