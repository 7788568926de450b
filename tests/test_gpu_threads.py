"""Several host threads, each with a context and a stream of its own, work on
datasets of different genome counts at once: launches whose shared memory grows
with the genomes must not depend on what another thread launches meanwhile."""
import threading

import numpy as np
import pytest

from paper_2510_23679_gb300 import pd, synth

pytestmark = pytest.mark.gpu

LETTERS = np.frombuffer(synth.ALPHABET, np.uint8)


def dataset(genomes, genes, seed):
    """Genomes of short mutated copies of a few families."""
    rng = np.random.default_rng(seed)
    family = LETTERS[rng.integers(0, 20, (7, 20))]
    out = []
    for _ in range(genomes):
        genome = []
        for _ in range(genes):
            gene = family[rng.integers(0, 7)].copy()
            gene[rng.integers(0, 20, 3)] = LETTERS[rng.integers(0, 20, 3)]
            genome.append(gene.tobytes())
        out.append(genome)
    return synth.from_strings(out)


def whole_run(ctx, ds):
    prof = pd.pd_build_profiles(ctx, ds.residues, ds.gene_ptr, ds.genome_ptr, 5)
    out = []
    for hits in (pd.pd_best_hits_all(ctx, prof), pd.pd_best_hits_all_filtered(ctx, prof, (1, 2), (1, 20)),
                 pd.pd_best_hits_shard(ctx, prof, 0, 2)):
        out += [*pd.pd_hits_copy(ctx, hits), pd.pd_bbh_copy(ctx, pd.pd_bbh_all(ctx, prof, hits))]
    return out


def test_contexts_of_several_threads():
    # genome counts on both sides of every layout of the tiers and row tiles
    data = [dataset(*shape) for shape in ((3, 9, 1), (60, 3, 2), (300, 2, 3), (700, 1, 4))]
    want = [whole_run(pd.pd_ctx_create(0), ds) for ds in data]
    failures = []
    start = threading.Barrier(len(data))

    def work(i):
        import torch
        try:
            stream = torch.cuda.Stream()
            ctx = pd.pd_ctx_create(0, stream=stream)
            start.wait(60)
            for _ in range(60):
                got = whole_run(ctx, data[i])
                if not all(np.array_equal(x, y) for x, y in zip(got, want[i])):
                    failures.append((i, "other results"))
            stream.synchronize()
        except Exception as e:  # reported by the main thread
            failures.append((i, repr(e)))

    threads = [threading.Thread(target=work, args=(i,)) for i in range(len(data))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not failures, failures[:4]
