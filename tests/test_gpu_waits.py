"""A look-back wait that is given up (index sort, prefix sums): the call fails
with PD_ERR_INTERNAL, no later pass touches what was not written, and the GPU
context stays usable.

The library's wait limit is a constant, so the two files that wait are compiled
once more with a limit of no polls: a tile whose predecessor is not ready at the
first look gives up.  A child process loads that library.  Whether a given wait
is given up depends on timing; a call that meets none must return the right
result."""
import glob
import json
import os
import subprocess
import sys

import pytest

from paper_2510_23679_gb300 import _build

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
WAITING = ("k_index.cu", "k_scan.cu")

CHILD = r"""
import json, sys
import numpy as np
from paper_2510_23679_gb300 import _build, pd, synth
_build.LIB = sys.argv[1]
pd.load(build=False)
import torch

LETTERS = np.frombuffer(synth.ALPHABET, np.uint8)


def dataset(seed, genes, length, genomes):
    rng = np.random.default_rng(seed)
    family = LETTERS[rng.integers(0, 20, (max(genes // 3, 1), length))]
    residues = family[rng.integers(0, len(family), genes)]
    other = rng.random(residues.shape) < 0.1
    residues[other] = LETTERS[rng.integers(0, 20, int(other.sum()))]
    return (np.ascontiguousarray(residues.reshape(-1)), np.arange(genes + 1, dtype=np.int64) * length,
            np.linspace(0, genes, genomes + 1).astype(np.int32))


def calls(ctx, data, k):
    prof = pd.pd_build_profiles(ctx, *data, k)
    yield "build", [pd.pd_profiles_get_info(prof).n_entries]
    yield "index", pd.pd_profiles_copy_index(ctx, prof)
    yield "vectors", pd.pd_profiles_copy_mv(ctx, prof)
    hits = pd.pd_best_hits_all(ctx, prof)
    yield "all", (*pd.pd_hits_copy(ctx, hits), pd.pd_bbh_copy(ctx, pd.pd_bbh_all(ctx, prof, hits)))
    hits = pd.pd_paralog_hits(ctx, prof)
    yield "paralogs", (*pd.pd_hits_copy(ctx, hits), pd.pd_bbh_copy(ctx, pd.pd_paralog_bbh(ctx, prof, hits)))
    yield "pair", pd.pd_bbh_copy(ctx, pd.pd_bbh(ctx, prof, 0, 1))
    jobs = np.array([[0, 1], [1, 2], [0, 2]], np.uint32)
    batch = pd.pd_bbh_pairs(ctx, prof, jobs)
    yield "pairs", (*pd.pd_batch_copy_hits(ctx, batch), *pd.pd_batch_copy_bbh(ctx, batch))
    a = np.arange(1000, dtype=np.uint32)
    yield "similarity", pd.pd_summin_list(ctx, prof, a, a[::-1].copy())
    batch = pd.pd_bbh_batch(ctx, *data, jobs[:1], np.array([k], np.int32))
    yield "batch", (*pd.pd_batch_copy_hits(ctx, batch), *pd.pd_batch_copy_bbh(ctx, batch))


def digest(x):
    import hashlib
    h = hashlib.sha256()
    for part in x:
        h.update(np.ascontiguousarray(np.asarray(part)).tobytes())
    return h.hexdigest()


out = []
# many tiles of windows; few windows but several tiles of genes (the prefix sums)
for seed, genes, length, genomes, repeat in ((1, 12000, 300, 4, 3), (2, 24000, 7, 4, 12), (3, 5000, 6, 3, 12)):
    data = dataset(seed, genes, length, genomes)
    for _ in range(repeat):
        ctx = pd.pd_ctx_create(0)
        it = calls(ctx, data, 5)
        while True:
            try:
                name, value = next(it)
                out.append([seed, name, digest(value)])
            except StopIteration:
                break
            except pd.PdError as e:
                out.append([seed, str(e), None, e.status])
                break
        del it
torch.cuda.synchronize()
assert int(torch.ones(1000, device="cuda").sum()) == 1000
print("RESULT", json.dumps(out))
"""


def run_child(lib):
    env = dict(os.environ, PYTHONPATH=ROOT)
    r = subprocess.run([sys.executable, "-c", CHILD, lib], capture_output=True, text=True, timeout=300, env=env, cwd=ROOT)
    assert r.returncode == 0, r.stderr[-2000:]
    return json.loads(r.stdout.split("RESULT ")[1])


def test_waits_given_up(tmp_path):
    lib = _build.build()
    want = {(r[0], r[1]): r[2] for r in run_child(lib)}
    assert all(v is not None for v in want.values()) and len(want) == 27
    objs = [o for o in glob.glob(os.path.join(_build.OUT_DIR, "*.cu.o")) if os.path.basename(o)[:-2] not in WAITING]
    for name in WAITING:
        objs.append(str(tmp_path / (name + ".o")))
        subprocess.run([_build._nvcc(), *_build.ARCH, *_build.NVCC_FLAGS, "-DPD_MAX_POLLS=0", "-c",
                        os.path.join(_build.CSRC, name), "-o", objs[-1]], check=True)
    hasty = str(tmp_path / "libpandelos_hasty.so")
    subprocess.run([_build._nvcc(), *_build.ARCH, "-shared", "-o", hasty, *objs], check=True)
    got = run_child(hasty)
    given_up = [r for r in got if r[2] is None]
    assert given_up, "no wait was given up"
    for r in got:
        if r[2] is None:
            assert r[3] == 10, r  # PD_ERR_INTERNAL
        else:
            assert want[(r[0], r[1])] == r[2], r
