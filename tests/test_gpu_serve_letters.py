"""pd_index_submit accepts exactly the amino-acid letters, wherever they stand
(the check takes 64 bytes at a time, then the rest one by one)."""
import numpy as np
import pytest

from paper_2510_23679_gb300 import pd, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("length,at", [(1, 0), (63, 62), (64, 0), (64, 63), (65, 64), (200, 127), (200, 128), (200, 199)])
def test_letters(length, at):
    ctx = pd.pd_ctx_create(0)
    ds = synth.from_strings([[b"ACDEFGHIKLMNPQRSTVWY"]])
    index = pd.pd_index_create(ctx, ds.residues, ds.gene_ptr, ds.genome_ptr, 3, 4 << 30)
    pd.pd_index_hold(index, True)
    for byte in range(256):
        res = np.frombuffer(synth.ALPHABET, np.uint8)[np.arange(length) % 20].copy()
        res[at] = byte
        if byte in synth.ALPHABET:
            assert pd.pd_index_submit(index, res, np.array([0, length], np.int64)) > 0
        else:
            with pytest.raises(pd.PdError) as e:
                pd.pd_index_submit(index, res, np.array([0, length], np.int64))
            assert e.value.status == 2, byte
    index.free()
