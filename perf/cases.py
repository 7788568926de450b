"""What the speed of this package is measured on.

The cases are the calls that a user of the package makes, over the sizes that
its configurations, tests and benchmark use: whole all-against-all runs from
four genomes to two hundred (from residues on the device, and from and to host
arrays), the nucleotide alphabet, queries on a profiled dataset (one genome
pair, many pairs, filtered and within-genome Best Hits, the similarity of
listed gene pairs), a batch of independent genome pairs, and a served index
that answers a burst of new genomes.

Inputs are pangenomes of mutated gene families: the model of the package's
`synth` module (core and accessory families, paralog copies, singletons,
substitutions and single-residue indels), drawn on the GPU so that the largest
takes well under a second.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2510_23679_gb300 import pd, synth

# Length distributions of genes: (median, sigma, shortest, longest) of a
# clipped log-normal, as in the package's workloads.
AMINO = (300, 0.5, 30, 2500)
AMINO_LONG = (900, 0.5, 30, 2500)
NUCLEOTIDE = (900, 0.5, 90, 7500)


# ---------------------------------------------------------------- the cases
def listed():
    return [
        # A handful of small genomes, profiled and compared: the smallest
        # whole run, bound by launches and host round trips.
        {"name": "all_4x250", "kind": "all", "genomes": 4, "genes": 250, "families": 200, "core": 0.0},
        # The ordinary whole run: one species' genomes.
        {"name": "all_50x3000", "kind": "all", "genomes": 50, "genes": 3000, "families": 4000, "core": 0.4},
        # The largest whole run of the benchmark: 200 genomes, 19,900 pairs.
        {"name": "all_200x4000", "kind": "all", "genomes": 200, "genes": 4000, "families": 12000, "core": 0.25},
        # Gene nucleotide sequences instead of proteins.
        {"name": "nucleotide_8x600", "kind": "nucleotide", "genomes": 8, "genes": 600, "families": 800, "core": 0.4},
        # An analysis script: host arrays in, Best Hits, BBH pairs and gene
        # families back in host arrays.
        {"name": "script_23x1700", "kind": "script", "genomes": 23, "genes": 1700, "families": 2300, "core": 0.4},
        # One genome pair of a profiled dataset: the smallest query.
        {"name": "pair_of_50x3000", "kind": "pair", "genomes": 50, "genes": 3000, "families": 4000, "core": 0.4},
        # Many listed genome pairs of one profiled dataset.
        {"name": "pairs_300_of_60x3000", "kind": "pairs", "genomes": 60, "genes": 3000, "families": 4000, "core": 0.4,
         "jobs": 300},
        # Best Hits under the length and shared-occurrence thresholds.
        {"name": "filtered_30x2000", "kind": "filtered", "genomes": 30, "genes": 2000, "families": 2700, "core": 0.4},
        # Paralogs: Best Hits and mutual pairs inside each genome.
        {"name": "paralogs_60x3000", "kind": "paralogs", "genomes": 60, "genes": 3000, "families": 4000, "core": 0.4},
        # The exact similarity of a candidate list of gene pairs.
        {"name": "listed_similarity_40x2500", "kind": "similarity", "genomes": 40, "genes": 2500, "families": 3300,
         "core": 0.4, "pairs": 1000003},
        # Independent two-genome problems, each at its own k, in one call.
        {"name": "batch_32", "kind": "batch", "jobs": 32, "genes_low": 500, "genes_high": 6000},
        # A service: opens an index on its resident genomes and answers a
        # burst of incoming ones.
        {"name": "served_4_on_30x3000", "kind": "served", "genomes": 30, "genes": 3000, "families": 4000, "core": 0.4,
         "incoming": 4, "genes_low": 1000, "genes_high": 7000},
    ]


def draw(rng):
    def spread(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["all", "all", "all", "nucleotide", "script", "pair", "pairs", "filtered", "paralogs",
                       "similarity", "batch", "served"])
    if kind == "batch":
        low = spread(100, 1500)
        return {"kind": kind, "jobs": spread(3, 60), "genes_low": low, "genes_high": low * rng.randint(2, 5)}
    most_genomes, most_genes = {"all": (200, 4000), "nucleotide": (24, 1500), "script": (40, 2500),
                                "pair": (60, 4000), "pairs": (80, 4000), "filtered": (50, 3000),
                                "paralogs": (80, 4000), "similarity": (50, 3000), "served": (40, 3500)}[kind]
    genes = spread(150, most_genes)
    case = {"kind": kind, "genomes": spread(3, most_genomes), "genes": genes,
            "families": max(40, int(genes * rng.uniform(0.8, 3.0))), "core": round(rng.choice([0.0, 0.25, 0.4]), 2)}
    if kind == "pairs":
        case["jobs"] = min(spread(10, 500), case["genomes"] * (case["genomes"] - 1))
    if kind == "similarity":
        case["pairs"] = spread(1000, 2000000)
    if kind == "served":
        case.update(incoming=rng.randint(1, 6), genes_low=genes // 3, genes_high=genes * 2)
    return case


# ---------------------------------------------------------------- inputs
def _letters(gen, n, alphabet):
    """n letter codes of the alphabet's background composition."""
    p = torch.tensor(synth.BACKGROUND if alphabet == 20 else synth.NT_BACKGROUND, device="cuda", dtype=torch.float32)
    edges = torch.cumsum(p, 0)[:-1].contiguous()
    return torch.bucketize(torch.rand(n, device="cuda", generator=gen), edges, right=True).to(torch.uint8)


def _lengths(rng, n, dist):
    median, sigma, lo, hi = dist
    return np.clip(np.rint(rng.lognormal(np.log(median), sigma, n)), lo, hi).astype(np.int64)


def _gene_families(rng, count, n_families, core):
    """Family of each gene of one genome (-1: a singleton of its own): the
    core families, accessory families, 10% paralog copies, 5% singletons."""
    n_single, n_copies = round(0.05 * count), round(0.10 * count)
    n_core = min(round(core * n_families), count - n_single)
    n_accessory = max(0, min(n_families - n_core, count - n_single - n_copies - n_core))
    held = np.concatenate([np.arange(n_core), n_core + rng.permutation(n_families - n_core)[:n_accessory]])
    copies = rng.choice(held, max(0, count - n_single - len(held)))
    return rng.permutation(np.concatenate([held, copies, np.full(n_single, -1)]))


def _pangenome(seed, counts, n_families, core, dist=AMINO, alphabet=20):
    """(residues uint8, gene_ptr int64, genome_ptr int32) on the device, and
    the family of each gene (host)."""
    rng = np.random.default_rng(seed)
    gen = torch.Generator("cuda").manual_seed(seed)
    family_len = _lengths(rng, n_families, dist)
    subst = torch.tensor(rng.uniform(0.0, 0.30, n_families + 1), device="cuda", dtype=torch.float32)
    indel = torch.tensor(rng.uniform(0.0, 0.05, n_families + 1), device="cuda", dtype=torch.float32)
    subst[-1] = indel[-1] = 0.0  # singletons are fresh sequences
    family = np.concatenate([_gene_families(rng, int(c), n_families, core) for c in counts])
    single = family < 0
    source_len = np.where(single, 0, family_len[family])
    source_len[single] = _lengths(rng, int(single.sum()), dist)
    ancestors = _letters(gen, int(family_len.sum()), alphabet)
    family_start = np.concatenate([[0], np.cumsum(family_len)])[:-1]

    length = torch.tensor(source_len, device="cuda")
    gene = torch.repeat_interleave(torch.arange(len(family), device="cuda", dtype=torch.int32), length)
    ends = torch.cumsum(length, 0)
    shift = torch.tensor(np.where(single, 0, family_start[family]), device="cuda") - (ends - length)
    of = torch.tensor(family, device="cuda")[gene]
    n = gene.numel()
    fresh = _letters(gen, n, alphabet)
    at = (torch.arange(n, device="cuda") + shift[gene]).clamp_(0, ancestors.numel() - 1)
    replaced = (torch.rand(n, device="cuda", generator=gen) < subst[of]) | (of < 0)
    code = torch.where(replaced, fresh, ancestors[at])
    del at, fresh, replaced
    u, rate = torch.rand(n, device="cuda", generator=gen), indel[of]
    repeats = (1 - (u < 0.5 * rate).to(torch.int64)) + ((u >= 0.5 * rate) & (u < rate)).to(torch.int64)
    del u, rate, of
    last = torch.cumsum(repeats, 0)
    code = torch.repeat_interleave(code, repeats)
    inserted = last[repeats == 2] - 1  # the second copy of an inserted position is a new letter
    code[inserted] = _letters(gen, inserted.numel(), alphabet)
    gene_ptr = torch.zeros(len(family) + 1, dtype=torch.int64, device="cuda")
    gene_ptr[1:] = last[ends - 1]
    table = torch.tensor(list(synth.ALPHABET if alphabet == 20 else synth.NT_ALPHABET), device="cuda", dtype=torch.uint8)
    genome_ptr = torch.tensor(np.concatenate([[0], np.cumsum(counts)]).astype(np.int32), device="cuda")
    return table[code.to(torch.int32)], gene_ptr, genome_ptr, family


def _join(parts):
    """Datasets one after the other."""
    residues = torch.cat([p[0] for p in parts])
    gene_ptr, genome_ptr = [parts[0][1][:1]], [parts[0][2][:1]]
    n_res = n_genes = 0
    for res, genes, genomes, _ in parts:
        gene_ptr.append(genes[1:] + n_res)
        genome_ptr.append(genomes[1:] + n_genes)
        n_res, n_genes = n_res + res.numel(), n_genes + genes.numel() - 1
    return residues, torch.cat(gene_ptr), torch.cat(genome_ptr)


def _k(n_residues, alphabet=20):
    """The k rule: the smallest k with alphabet^k >= the residues."""
    k = 1
    while alphabet ** k < n_residues:
        k += 1
    return k


def _gene_counts(case):
    """Genes of each genome: a case's own, whatever the seed of its inputs."""
    rng = np.random.default_rng(case.get("genomes", 0) * 100003 + case.get("genes", 0) + case.get("jobs", 0))
    if case["kind"] == "batch":
        return rng.integers(case["genes_low"], case["genes_high"] + 1, 2 * case["jobs"])
    counts = np.maximum(rng.poisson(case["genes"], case["genomes"]), 20)
    if case["kind"] == "served":
        counts = np.concatenate([counts, rng.integers(case["genes_low"], case["genes_high"] + 1, case["incoming"])])
    return counts


def _one_pair(case):
    n = case["genomes"]
    return n // 2 + 1 - n % 2, n // 4  # two different genomes, the later one first


def _genome_pairs(case):
    """Ordered pairs of different genomes, each at most once."""
    n = case["genomes"]
    chosen = np.random.default_rng(case["jobs"]).choice(n * (n - 1), case["jobs"], replace=False)
    return np.stack([chosen // (n - 1), (chosen // (n - 1) + 1 + chosen % (n - 1)) % n], 1).astype(np.uint32)


def _input(case, seed):
    """Everything `prepare` and `exact` start from, from the seed alone."""
    rng = np.random.default_rng(seed + 1)
    kind = case["kind"]
    counts = _gene_counts(case)
    if kind == "batch":
        parts = []
        for j in range(case["jobs"]):
            of_job = counts[2 * j:2 * j + 2]
            parts.append(_pangenome(seed * 1000 + j, of_job, int(math.ceil(int(of_job.max()) * 4 / 3)), 0.4,
                                    AMINO_LONG if j % 2 else AMINO))
        residues, gene_ptr, genome_ptr = _join(parts)
        return {"residues": residues, "gene_ptr": gene_ptr, "genome_ptr": genome_ptr,
                "jobs": np.arange(2 * case["jobs"], dtype=np.uint32).reshape(-1, 2),
                "job_k": np.array([_k(p[0].numel()) for p in parts], np.int32)}
    alphabet = 4 if kind == "nucleotide" else 20
    residues, gene_ptr, genome_ptr, family = _pangenome(seed, counts, case["families"], case["core"],
                                                        NUCLEOTIDE if alphabet == 4 else AMINO, alphabet)
    given = {"residues": residues, "gene_ptr": gene_ptr, "genome_ptr": genome_ptr, "alphabet": alphabet,
             "k": _k(residues.numel(), alphabet)}
    if kind == "pair":
        given["pair"] = _one_pair(case)
    if kind == "pairs":
        given["jobs"] = _genome_pairs(case)
    if kind == "filtered":
        given["theta"], given["tau"] = (1, 2), (1, 20)
    if kind == "similarity":
        # candidate pairs as a clustering gives them: mostly genes of one family
        by_family = np.argsort(family, kind="stable")
        at = rng.integers(0, len(by_family), case["pairs"])
        other = (at + rng.integers(1, 2 * case["genomes"], case["pairs"])) % len(by_family)
        given["a"] = torch.tensor(by_family[at].astype(np.int32), device="cuda")
        given["b"] = torch.tensor(by_family[other].astype(np.int32), device="cuda")
    if kind == "served":
        n = case["genomes"]
        first_gene = int(genome_ptr[n])
        starts = gene_ptr[genome_ptr.long()].tolist()
        given["resident"] = (residues[:starts[n]], gene_ptr[:first_gene + 1], genome_ptr[:n + 1])
        given["k"] = _k(starts[n])
        given["incoming"] = []
        for i in range(n, n + case["incoming"]):
            genes = gene_ptr[int(genome_ptr[i]):int(genome_ptr[i + 1]) + 1]
            given["incoming"].append((residues[starts[i]:starts[i + 1]].cpu().numpy(),
                                      (genes - starts[i]).cpu().numpy()))
    return given


def _results(case):
    """The buffers that a program keeps for results: entries of each by name.
    Best Hits hold one target gene per query gene and genome, ties more, so a
    program makes room for a few more than that."""
    kind, counts = case["kind"], _gene_counts(case)
    genes, others = int(counts.sum()), case.get("genomes", 2) - 1
    if kind == "batch":
        hits, rows = genes, genes
    elif kind == "pairs":
        rows = int(counts[_genome_pairs(case).astype(np.int64)].sum())
        hits = rows
    elif kind == "pair":
        rows = int(counts[_one_pair(case)[0]])
        hits = rows
    elif kind == "paralogs":
        hits, rows = genes, genes
    else:
        hits, rows = genes * others, genes
    hits = hits + hits // 2 + 4096
    sizes = {"row_ptr": rows + 1, "cols": hits, "s": hits, "bbh_a": hits // 2, "bbh_b": hits // 2}
    if kind in ("batch", "pairs"):
        sizes["job_ptr"] = case["jobs"] + 1
    return sizes


def _buffers(sizes, **where):
    return {name: torch.zeros(n, dtype=torch.int64 if name.endswith("ptr") else torch.int32, **where)
            for name, n in sizes.items()}


def prepare(case, seed):
    given = _input(case, seed)
    kind = case["kind"]
    state = {"kind": kind, "ctx": pd.pd_ctx_create(0), **given}
    data = (given["residues"], given["gene_ptr"], given["genome_ptr"])
    if kind == "script":
        state["host"] = tuple(x.cpu().pin_memory() for x in data)
        state["results"] = _buffers(_results(case), pin_memory=True)
    elif kind == "served":
        state["budget"] = 40 << 30
        state["results"] = []
        for _, gene_ptr in given["incoming"]:
            n = (len(gene_ptr) - 1) * case["genomes"]
            sizes = {"row_ptr": len(gene_ptr), "cols": n + n // 2 + 4096, "s": n + n // 2 + 4096, "bbh": n + 4096}
            state["results"].append({name: np.zeros((m, 2) if name == "bbh" else m,
                                                    np.int64 if name == "row_ptr" else np.int32)
                                     for name, m in sizes.items()})
    elif kind != "similarity":
        state["results"] = _buffers(_results(case), device="cuda")
    if kind in ("pair", "pairs", "filtered", "paralogs", "similarity"):
        state["profiles"] = pd.pd_build_profiles(state["ctx"], *data, given["k"])
    return state


# ---------------------------------------------------------------- one pass
def _check_room(results, n_hits, n_bbh):
    if n_hits > len(results["cols"]) or n_bbh > len(results["bbh_a"]):
        raise RuntimeError(f"{n_hits} Best Hits or {n_bbh} BBH pairs do not fit the result buffers")


def _copy(ctx, results, hits, bbh):
    """Best Hits (CSR with sum-min values) and BBH pairs into the program's buffers."""
    _check_room(results, pd.pd_hits_get_info(hits).n_hits, pd.pd_bbh_count(bbh))
    pd.pd_hits_copy(ctx, hits, results["row_ptr"], results["cols"], results["s"])
    pd.pd_bbh_copy(ctx, bbh, results["bbh_a"], results["bbh_b"])
    return results


def _copy_batch(ctx, results, batch):
    info = pd.pd_batch_get_info(batch)
    _check_room(results, info.n_hits, info.n_bbh)
    pd.pd_batch_copy_hits(ctx, batch, results["row_ptr"], results["cols"], results["s"])
    pd.pd_batch_copy_bbh(ctx, batch, results["job_ptr"], results["bbh_a"], results["bbh_b"])
    return results


def _serve(state):
    """Opens an index on the resident genomes and answers the incoming ones,
    which arrive together (admission is held until all are queued, so every
    answer is against the resident genomes)."""
    index = pd.pd_index_create(state["ctx"], *state["resident"], state["k"], state["budget"])
    pd.pd_index_hold(index, True)
    tickets = [pd.pd_index_submit(index, *genome) for genome in state["incoming"]]
    pd.pd_index_hold(index, False)
    for ticket, results in zip(tickets, state["results"]):
        answer = pd.pd_reply_copy(pd.pd_index_poll(index, ticket))
        for name, part in zip(("row_ptr", "cols", "s", "bbh"), answer):
            results[name][:len(part)] = part
    index.free()
    return state["results"]


def run(state):
    kind, ctx = state["kind"], state["ctx"]
    if kind in ("all", "nucleotide"):
        profiles = pd.pd_build_profiles_alphabet(ctx, state["residues"], state["gene_ptr"], state["genome_ptr"],
                                                 state["alphabet"], state["k"])
        hits = pd.pd_best_hits_all(ctx, profiles)
        return _copy(ctx, state["results"], hits, pd.pd_bbh_all(ctx, profiles, hits))
    if kind == "script":
        profiles = pd.pd_build_profiles(ctx, *state["host"], state["k"])
        hits = pd.pd_best_hits_all(ctx, profiles)
        bbh = pd.pd_bbh_all(ctx, profiles, hits)
        family, n_families = pd.pd_families(ctx, bbh, state["host"][1].numel() - 1)
        return {**_copy(ctx, state["results"], hits, bbh), "family": family, "n_families": n_families}
    if kind == "pair":
        hits = pd.pd_best_hits(ctx, state["profiles"], *state["pair"])
        return _copy(ctx, state["results"], hits, pd.pd_bbh(ctx, state["profiles"], *state["pair"]))
    if kind == "pairs":
        return _copy_batch(ctx, state["results"], pd.pd_bbh_pairs(ctx, state["profiles"], state["jobs"]))
    if kind == "filtered":
        hits = pd.pd_best_hits_all_filtered(ctx, state["profiles"], state["theta"], state["tau"])
        return _copy(ctx, state["results"], hits, pd.pd_bbh_all(ctx, state["profiles"], hits))
    if kind == "paralogs":
        hits = pd.pd_paralog_hits(ctx, state["profiles"])
        return _copy(ctx, state["results"], hits, pd.pd_paralog_bbh(ctx, state["profiles"], hits))
    if kind == "similarity":
        s, den = torch.empty_like(state["a"]), torch.empty_like(state["a"])
        pd.pd_summin_list(ctx, state["profiles"], state["a"], state["b"], s, den)
        return {"s": s, "den": den}
    if kind == "batch":
        return _copy_batch(ctx, state["results"],
                           pd.pd_bbh_batch(ctx, state["residues"], state["gene_ptr"], state["genome_ptr"],
                                           state["jobs"], state["job_k"]))
    if kind == "served":
        return _serve(state)
    raise ValueError(f"unknown kind of case: {kind}")


# ---------------------------------------------------------------- work
def work(case):
    """The inputs of the call (residues and offsets, or the k-mer vectors of
    the genes that a profiled dataset's query compares) read once and the
    results written once; sizes that depend on the data are expected values of
    the model.  The arithmetic is on integers (no floating point): flops 0."""
    kind = case["kind"]
    mean = (900 if kind == "nucleotide" else 300) * math.exp(0.125)
    entry = 6.0  # one k-mer of a gene's vector: its id and its count
    pair_hits = 0.95  # Best Hits per query gene and target genome
    pair_bbh = 0.35  # BBH pairs per gene and other genome
    if kind == "batch":
        genes = case["jobs"] * (case["genes_low"] + case["genes_high"])
        residues = genes * 0.5 * (300 + 900) * math.exp(0.125)
        return {"bytes": residues + 8.0 * genes + genes * (8 + 8 * pair_hits + 8 * pair_bbh), "flops": 0.0}
    genes, others = case["genomes"] * case["genes"], case["genomes"] - 1
    if kind in ("all", "nucleotide", "script"):
        return {"bytes": genes * (mean + 8 + 8 + others * 8 * (pair_hits + pair_bbh)), "flops": 0.0}
    if kind == "pair":
        genes = 2 * case["genes"]
        return {"bytes": genes * (mean * entry + 8 + 8 * (pair_hits + pair_bbh)), "flops": 0.0}
    if kind == "pairs":
        rows = case["jobs"] * 2 * case["genes"]
        return {"bytes": genes * mean * entry + rows * (8 + 8 * (pair_hits + pair_bbh)), "flops": 0.0}
    if kind == "filtered":
        return {"bytes": genes * (mean * entry + 8 + others * 8 * 0.8), "flops": 0.0}
    if kind == "paralogs":
        return {"bytes": genes * (mean * entry + 8 + 8 * 1.2), "flops": 0.0}
    if kind == "similarity":
        return {"bytes": genes * mean * entry + case["pairs"] * 16.0, "flops": 0.0}
    incoming = case["incoming"] * 0.5 * (case["genes_low"] + case["genes_high"])
    return {"bytes": (genes + incoming) * (mean + 8) + incoming * (8 + case["genomes"] * 8 * (pair_hits + pair_bbh)),
            "flops": 0.0}


# ---------------------------------------------------------------- exact results
_MOST_SHARED = 400_000_000  # shared k-mers counted pair by pair below


class _Shared:
    """Every pair of genes that share a k-mer, a before b, with its sum of
    minima s (Eq. (5)) and the occurrences of the shared k-mers on each side
    (Eq. (7)); `windows` per gene; None in `s` if there are too many."""

    def __init__(self, residues, gene_ptr, k, alphabet, segment=None):
        letters = synth.ALPHABET if alphabet == 20 else synth.NT_ALPHABET
        number = torch.zeros(256, dtype=torch.int64, device="cuda")
        number[torch.tensor(list(letters), device="cuda")] = torch.arange(alphabet, device="cuda")
        digit = number[residues.int()]
        n, G = digit.numel(), gene_ptr.numel() - 1
        length = gene_ptr[1:] - gene_ptr[:-1]
        self.windows = (length - k + 1).clamp_(min=0)
        gene = torch.repeat_interleave(torch.arange(G, device="cuda"), length)
        code = torch.zeros(n - k + 1, dtype=torch.int64, device="cuda")
        for t in range(k):
            code = code * alphabet + digit[t:n - k + 1 + t]
        if segment is not None:
            code += segment[gene[:n - k + 1]] * alphabet ** k
        inside = torch.arange(n - k + 1, device="cuda") + k <= gene_ptr[1:][gene[:n - k + 1]]
        key, count = torch.unique(code[inside] * G + gene[:n - k + 1][inside], return_counts=True)
        del digit, code, inside
        code, gene = key // G, key % G
        _, size = torch.unique_consecutive(code, return_counts=True)
        behind = torch.repeat_interleave(torch.cumsum(size, 0), size) - torch.arange(code.numel(), device="cuda") - 1
        self.s = None
        if int(behind.sum()) > _MOST_SHARED:
            return
        i = torch.repeat_interleave(torch.arange(code.numel(), device="cuda"), behind)
        first = torch.cumsum(behind, 0) - behind
        j = i + 1 + torch.arange(i.numel(), device="cuda") - first[i]
        pair, where = torch.unique(gene[i] * G + gene[j], return_inverse=True)
        self.a, self.b = pair // G, pair % G
        self.s, self.occ_a, self.occ_b = (torch.zeros_like(pair).index_add_(0, where, x) for x in (
            torch.minimum(count[i], count[j]), count[i], count[j]))


def _best(a, b, s, group, windows):
    """The pairs (a, b) with the largest s / (La + Lb - s) of their group,
    ascending by (a, b): 64-bit quotients of integers below 2^17 are equal
    exactly when the ratios are."""
    ratio = s.double() / (windows[a] + windows[b] - s).double()
    ids, group = torch.unique(group, return_inverse=True)
    best = torch.zeros(ids.numel(), dtype=torch.float64, device="cuda").scatter_reduce_(0, group, ratio, "amax")
    keep = (ratio == best[group]).nonzero().flatten()
    return keep[torch.argsort(a[keep] * (1 << 32) + b[keep])]


def _rows(a, n_rows):
    row_ptr = torch.zeros(n_rows + 1, dtype=torch.int64, device="cuda")
    row_ptr[1:] = torch.cumsum(torch.bincount(a, minlength=n_rows), 0)
    return row_ptr


def _mutual(a, b, n):
    """The pairs (a, b) that are there as (b, a) too, with a < b."""
    key = a * n + b
    keep = torch.isin(key, b * n + a) & (a < b)
    return a[keep], b[keep]


def _padded(case, **out):
    """The results at the start of zeroed buffers, as `run` leaves them."""
    sizes = _results(case)
    return {name: torch.cat([x, x.new_zeros(sizes[name] - x.numel())]) if name in sizes else x for name, x in out.items()}


def exact(case, seed):
    kind = case["kind"]
    given = _input(case, seed)
    gene_ptr, genome_ptr = given["gene_ptr"], given["genome_ptr"].long()
    G = gene_ptr.numel() - 1
    genome = torch.repeat_interleave(torch.arange(genome_ptr.numel() - 1, device="cuda"), genome_ptr.diff())
    k, segment, residues = given.get("k"), None, given["residues"]
    if kind == "served" or (kind == "batch" and len(set(given["job_k"].tolist())) > 1) or residues.numel() > 1 << 27:
        return None  # a service's answers and mixed k are compared with the plain calls in the tests
    if kind == "batch":
        k, segment = int(given["job_k"][0]), genome // 2
    shared = _Shared(residues, gene_ptr, k, given.get("alphabet", 20), segment)
    if shared.s is None:
        return None
    n = genome_ptr.numel() - 1
    if kind == "similarity":
        a, b = given["a"].long(), given["b"].long()
        key, want = shared.a * G + shared.b, torch.minimum(a, b) * G + torch.maximum(a, b)
        at = torch.searchsorted(key, want).clamp_(max=max(key.numel() - 1, 0))
        s = torch.where(key[at] == want, shared.s[at], torch.zeros_like(want))
        s = torch.where(a == b, shared.windows[a], s)
        return {"s": s, "den": shared.windows[a] + shared.windows[b] - s}
    keep = (genome[shared.a] == genome[shared.b]) == (kind == "paralogs")
    if kind == "filtered":
        (tn, td), (on, od) = given["theta"], given["tau"]
        la, lb = (shared.windows[x] + k - 1 for x in (shared.a, shared.b))
        keep &= (la * td >= tn * lb) & (lb * td >= tn * la)
        keep &= (shared.occ_a * od >= on * shared.windows[shared.a]) & (shared.occ_b * od >= on * shared.windows[shared.b])
    a, b, s = shared.a[keep], shared.b[keep], shared.s[keep]
    a, b, s = torch.cat([a, b]), torch.cat([b, a]), torch.cat([s, s])  # both directions
    at = _best(a, b, s, a * n + genome[b], shared.windows)
    a, b, s = a[at], b[at], s[at]
    if kind in ("all", "nucleotide", "filtered", "paralogs"):
        x, y = _mutual(a, b, G)
        return _padded(case, row_ptr=_rows(a, G), cols=b, s=s, bbh_a=x, bbh_b=y)
    if kind == "script":
        x, y = _mutual(a, b, G)
        family = torch.arange(G, device="cuda")
        while True:  # the smallest gene that a gene is linked to, until nothing changes
            low = family.clone().scatter_reduce_(0, x, family[y], "amin").scatter_reduce_(0, y, family[x], "amin")
            low = low[low]
            if torch.equal(low, family):
                break
            family = low
        return _padded(case, row_ptr=_rows(a, G), cols=b, s=s, bbh_a=x, bbh_b=y, family=family,
                       n_families=int(torch.unique(family).numel()))
    if kind == "pair":
        i, j = given["pair"]
        to = (genome[a] == i) & (genome[b] == j)
        both = to | ((genome[a] == j) & (genome[b] == i))
        # pairs are (gene of i, gene of j), whichever genome comes first
        x, y = _mutual(a[both], b[both], G)
        if i > j:
            x, y = y, x
        order = torch.argsort(x * G + y)
        n_rows = int(genome_ptr[i + 1] - genome_ptr[i])
        return _padded(case, row_ptr=_rows(a[to] - genome_ptr[i], n_rows), cols=b[to] - genome_ptr[j], s=s[to],
                       bbh_a=x[order] - genome_ptr[i], bbh_b=y[order] - genome_ptr[j])
    out = {name: [] for name in ("rows", "cols", "s", "job", "bbh_a", "bbh_b")}
    bounds = genome_ptr.tolist()
    first = torch.searchsorted(a, genome_ptr).tolist()  # hits of each genome's genes
    for i, j in given["jobs"].tolist():
        hits = []
        for p, q in ((i, j), (j, i)):
            to = torch.arange(first[p], first[p + 1], device="cuda")
            to = to[genome[b[to]] == q]
            hits.append((a[to], b[to]))
            out["rows"].append(torch.bincount(a[to] - bounds[p], minlength=bounds[p + 1] - bounds[p]))
            out["cols"].append(b[to] - bounds[q])
            out["s"].append(s[to])
        keep = torch.isin(hits[0][0] * G + hits[0][1], hits[1][1] * G + hits[1][0])
        out["bbh_a"].append(hits[0][0][keep] - bounds[i])
        out["bbh_b"].append(hits[0][1][keep] - bounds[j])
        out["job"].append(out["bbh_a"][-1].numel())
    rows = torch.cat(out["rows"])
    zero = torch.zeros(1, dtype=torch.int64, device="cuda")
    return _padded(case, row_ptr=torch.cat([zero, torch.cumsum(rows, 0)]), cols=torch.cat(out["cols"]),
                   s=torch.cat(out["s"]), bbh_a=torch.cat(out["bbh_a"]), bbh_b=torch.cat(out["bbh_b"]),
                   job_ptr=torch.tensor(np.concatenate([[0], np.cumsum(out["job"])]), device="cuda"))
