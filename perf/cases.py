"""The workloads whose speed is tracked: whole calls of the public entry points
of ``paper_1401_7457_gb300.binding``, from a few thousand suffixes to 808
million, as programs that build BWTs of read collections make them.

A case is one call (or one batch, or one burst of served requests) on seeded
reads: i.i.d. uniform bases, or reads drawn from both strands of a random
genome with 1% substitutions (optionally with 5% of 1 kb repeats).  The reads
are drawn on the GPU, so that inputs of every size are quick to make.
"""
import math

import numpy as np
import torch

from paper_1401_7457_gb300 import binding

BATCH_LENGTHS = (36, 76, 100, 150)
SERVE_LENGTHS = (100, 150)


def listed():
    return [
        # A few thousand reads inside a latency-bound loop that may not allocate
        # device memory: launches and host round trips are all there is.
        {"name": "noalloc-2k-76", "kind": "noalloc", "reads": 2_000, "length": 76, "genome": 0},
        # The smallest configuration: 10,000 random reads, device buffers.
        {"name": "tiny-10k-100", "kind": "build", "reads": 10_000, "length": 100, "genome": 0},
        # A bacterial genome at 20x on device buffers: the ordinary build.
        {"name": "genome-1M-100", "kind": "build", "reads": 1_000_000, "length": 100, "genome": 5_000_000},
        # The same collection through pinned host buffers: the end-to-end call.
        {"name": "host-1M-100", "kind": "host", "reads": 1_000_000, "length": 100, "genome": 5_000_000},
        # As many bases in longer reads (the read-length series' last point).
        {"name": "long-250k-400", "kind": "build", "reads": 250_000, "length": 400, "genome": 5_000_000},
        # Trimmed reads: lengths from 20 to 300 in one collection.
        {"name": "mixed-300k", "kind": "mixed", "reads": 300_000, "length": 300, "shortest": 20, "genome": 2_000_000},
        # A larger, repeat-rich genome at 50x whose packed reads exceed L2.
        {"name": "rich-8M-100", "kind": "build", "reads": 8_000_000, "length": 100, "genome": 16_000_000, "repeats": True},
        # The same kind of reads under a device budget of a third of the
        # workspace: built in slices, as a GPU shared with other work does.
        {"name": "sliced-5M-100", "kind": "sliced", "reads": 5_000_000, "length": 100, "genome": 10_000_000, "repeats": True,
         "slices": 3},
        # Many independent samples in one call, most of them small.
        {"name": "batch-20", "kind": "batch", "collections": 20, "least": 10_000, "most": 400_000, "spec": 4},
        # A burst of requests on a server with host buffers.
        {"name": "serve-12", "kind": "serve", "requests": 12, "least": 50_000, "most": 1_000_000, "spec": 5},
        # One of four bucket ranges of a collection: a rank's share of a
        # sharded build, or one round of a checkpointed one.
        {"name": "part-1M-100", "kind": "part", "reads": 1_000_000, "length": 100, "genome": 5_000_000, "parts": 4, "part": 1},
        # The BWT with the sorted suffix list, for callers that sample it.
        {"name": "sa-400k-150", "kind": "sa", "reads": 400_000, "length": 150, "genome": 2_000_000},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(("noalloc", "build", "build", "build", "host", "mixed", "sliced", "batch", "serve", "part", "sa"))
    if kind == "batch":
        return {"kind": kind, "collections": rng.randint(2, 20), "least": 10_000, "most": _log_int(rng, 20_000, 600_000),
                "spec": rng.randrange(1 << 30)}
    if kind == "serve":
        return {"kind": kind, "requests": rng.randint(1, 16), "least": 50_000, "most": _log_int(rng, 100_000, 1_500_000),
                "spec": rng.randrange(1 << 30)}
    if kind == "noalloc":
        length = rng.randint(30, 150)
        return {"kind": kind, "reads": _log_int(rng, 300, (1 << 21) // (length + 1)), "length": length, "genome": 0}
    length = rng.choice((36, 76, 100, 100, 150, 250, rng.randint(30, 400)))
    most = {"build": 800_000_000, "host": 200_000_000, "mixed": 100_000_000, "sliced": 500_000_000, "part": 200_000_000,
            "sa": 100_000_000}[kind] // (length + 1)
    least = {"build": 500, "host": 500, "mixed": 500, "sliced": 40_000_000 // (length + 1), "part": 10_000, "sa": 500}[kind]
    reads = _log_int(rng, least, most)
    case = {"kind": kind, "reads": reads, "length": length,
            "genome": 0 if rng.random() < 0.2 else max(2 * length + 10_000, int(reads * length / rng.uniform(15, 60)))}
    if kind == "mixed":
        case["shortest"] = rng.randint(10, length)
    if kind in ("build", "sliced") and case["genome"] > 1_000_000:
        case["repeats"] = rng.random() < 0.5
    if kind == "sliced":
        case["slices"] = rng.randint(2, 5)
    if kind == "part":
        case["parts"] = rng.randint(2, 8)
        case["part"] = rng.randrange(case["parts"])
    return case


# ---- inputs -------------------------------------------------------------------

def _generator(seed, salt=0):
    g = torch.Generator(device="cuda")
    g.manual_seed((seed * 1_000_003 + salt * 7_919 + 12_345) & 0x7FFFFFFFFFFFFFFF)
    return g


def _genome(size, g, repeats):
    """`size` random bases; with `repeats`, 5% of them copies (ten of each) of
    1,000-base templates with 0.5% substitutions."""
    genome = torch.randint(0, 4, (size,), generator=g, device="cuda", dtype=torch.uint8)
    if repeats:
        copies = size // 20_000
        slots = torch.randperm(size // 1_000, generator=g, device="cuda")[:copies]
        which = torch.randint(0, max(1, copies // 10), (copies,), generator=g, device="cuda")
        templates = torch.randint(0, 4, (max(1, copies // 10), 1_000), generator=g, device="cuda", dtype=torch.uint8)
        block = _substituted(templates[which], 0.005, g)
        at = slots[:, None] * 1_000 + torch.arange(1_000, device="cuda")[None, :]
        genome[at.reshape(-1)] = block.reshape(-1)
    return genome


def _substituted(block, rate, g):
    hit = torch.rand(block.shape, generator=g, device="cuda") < rate
    other = torch.randint(1, 4, block.shape, generator=g, device="cuda", dtype=torch.uint8)
    return torch.where(hit, (block + other) & 3, block)


def _packed(codes):
    """2-bit words of a flat array of base codes, first base in the top bits."""
    pad = (-codes.numel()) % 16
    if pad:
        codes = torch.cat([codes, torch.zeros(pad, dtype=torch.uint8, device=codes.device)])
    shifts = torch.arange(30, -2, -2, device=codes.device, dtype=torch.int64)
    return (codes.view(-1, 16).to(torch.int64) << shifts).sum(1).to(torch.int32)


def _blocks(reads, length, genome_size, repeats, g):
    """The reads, a block of rows of base codes at a time."""
    genome = _genome(genome_size, g, repeats) if genome_size else None
    col = torch.arange(length, device="cuda")
    step = max(16, (1 << 25) // length // 16 * 16)  # a multiple of 16 reads: every block fills whole words
    for r0 in range(0, reads, step):
        m = min(step, reads - r0)
        if genome is None:
            yield torch.randint(0, 4, (m, length), generator=g, device="cuda", dtype=torch.uint8)
            continue
        start = torch.randint(0, genome_size - length + 1, (m,), generator=g, device="cuda")
        block = genome[start[:, None] + col[None, :]]
        reverse = torch.rand((m, 1), generator=g, device="cuda") < 0.5
        block = torch.where(reverse, 3 - block.flip(1), block)
        yield _substituted(block, 0.01, g)


def _collection(reads, length, genome_size, repeats, g):
    """(packed words, lengths) on the GPU of reads of one length."""
    words = torch.cat([_packed(b.reshape(-1)) for b in _blocks(reads, length, genome_size, repeats, g)])
    return words, torch.full((reads,), length, dtype=torch.int32, device="cuda")


def _mixed_codes(case, seed):
    """(codes, lengths) on the GPU of reads of several lengths: whole reads cut
    to their first bases (the lengths are the case's, in the seed's order)."""
    g = _generator(seed)
    lens = torch.randint(case["shortest"], case["length"] + 1, (case["reads"],), generator=_generator(0), device="cuda")
    lens = lens[torch.randperm(case["reads"], generator=g, device="cuda")]
    col = torch.arange(case["length"], device="cuda")
    kept, at = [], 0
    for block in _blocks(case["reads"], case["length"], case["genome"], case.get("repeats", False), g):
        kept.append(block[col[None, :] < lens[at:at + block.shape[0], None]])
        at += block.shape[0]
    return torch.cat(kept), lens


def _specs(case):
    """(reads, length, genome) of every collection of a batch or a burst of requests."""
    rng = np.random.Generator(np.random.PCG64(case["spec"]))
    out = []
    batch = case["kind"] == "batch"
    for _ in range(case["collections"] if batch else case["requests"]):
        n = int(round(math.exp(rng.uniform(math.log(case["least"]), math.log(case["most"])))))
        lengths = BATCH_LENGTHS if batch else SERVE_LENGTHS
        length = int(lengths[int(rng.integers(0, len(lengths)))])
        coverage = float(rng.uniform(20.0, 50.0))
        out.append((n, length, min(max(int(n * length / coverage), 100_000), 20_000_000) if batch else 0))
    return out


def _outputs(reads, suffixes, where):
    kw = {"device": "cuda"} if where == "device" else {"pin_memory": True}
    return (torch.zeros((suffixes + 15) // 16, dtype=torch.int32, **kw), torch.zeros(reads, dtype=torch.int64, **kw),
            torch.zeros(5, dtype=torch.int64, **kw))


def _pinned(t):
    return t.cpu().pin_memory()


def prepare(case, seed):
    kind = case["kind"]
    if kind in ("batch", "serve"):
        items = []
        for j, (n, length, genome) in enumerate(_specs(case)):
            words, lens = _collection(n, length, genome, False, _generator(seed, j + 1))
            if kind == "serve":
                words, lens = _pinned(words), _pinned(lens)
            items.append((words, lens, *_outputs(n, n * (length + 1), "device" if kind == "batch" else "host")))
        handle = binding.Context(device=0) if kind == "batch" else binding.Server(device=0)
        torch.cuda.synchronize()
        return {"kind": kind, "items": items, "handle": handle}
    if kind == "mixed":
        codes, lens = _mixed_codes(case, seed)
        words, lens = _packed(codes), lens.to(torch.int32)
        suffixes = codes.numel() + case["reads"]
    else:
        words, lens = _collection(case["reads"], case["length"], case["genome"], case.get("repeats", False), _generator(seed))
        suffixes = case["reads"] * (case["length"] + 1)
    state = {"kind": kind, "words": words, "lens": lens}
    torch.cuda.synchronize()
    if kind == "noalloc":
        state["lens"] = lens.cpu().numpy().view(np.uint32)
        state["out"] = _outputs(case["reads"], suffixes, "device")
        return state
    budget = 0
    if kind == "sliced":
        # Room for the look-back words of every suffix and one slice's ids, keys and group lists.
        budget = int(6 << 20) + int(0.5 * suffixes + 17.25 * suffixes / case["slices"])
    state["ctx"] = binding.Context(device=0, budget_bytes=budget)
    if kind == "host":
        state["words"], state["lens"] = _pinned(words), _pinned(lens)
    if kind == "part":
        counts = state["ctx"].bucket_counts(words, lens)
        buckets, rows = binding.split_parts(counts, case["parts"])
        p = case["part"]
        state["range"] = (int(buckets[p]), int(buckets[p + 1]), int(rows[p]), int(rows[p + 1] - rows[p]))
        state["counts"] = counts
        # Buffers that hold any part of the collection: a rank allocates them before it knows its rows.
    state["out"] = _outputs(case["reads"], suffixes, "host" if kind == "host" else "device")
    if kind == "sa":
        state["sa"] = torch.zeros(suffixes, dtype=torch.int64, device="cuda")
    return state


def run(state):
    kind = state["kind"]
    if kind == "batch":
        state["handle"].build_batch(state["items"])
        return [item[2:] for item in state["items"]]
    if kind == "serve":
        tickets = [state["handle"].submit(*item) for item in state["items"]]
        for t in tickets:
            state["handle"].wait(t)
        return [item[2:] for item in state["items"]]
    bwt, dollar, counts = state["out"]
    if kind == "noalloc":
        binding.build_noalloc(state["words"], state["lens"], bwt, dollar, counts)
    elif kind == "part":
        lo, hi, row0, rows = state["range"]
        state["ctx"].build_part(state["words"], state["lens"], lo, hi, row0, rows, bwt, dollar, counts,
                                bucket_counts=state["counts"])
    elif kind == "sa":
        state["ctx"].build(state["words"], state["lens"], bwt, dollar, counts, out_sa=state["sa"])
        return state["out"] + (state["sa"],)
    else:
        state["ctx"].build(state["words"], state["lens"], bwt, dollar, counts)
    return state["out"]


def work(case):
    """The packed reads and their lengths read once, the packed BWT, the $ rows
    and the counts written once (and the suffix list, where asked for); sorting
    is not floating-point work."""
    if case["kind"] in ("batch", "serve"):
        sizes = [(n, n * length) for n, length, _ in _specs(case)]
    elif case["kind"] == "mixed":
        sizes = [(case["reads"], case["reads"] * (case["shortest"] + case["length"]) // 2)]
    else:
        sizes = [(case["reads"], case["reads"] * case["length"])]
    total = 0
    for n, bases in sizes:
        rows = bases + n
        written = rows // case["parts"] if case["kind"] == "part" else rows
        total += bases // 4 + 4 * n + written // 4 + 8 * n + 40 + (8 * rows if case["kind"] == "sa" else 0)
    return {"bytes": total, "flops": 0}


# ---- the same results from plain torch ------------------------------------------

def _sorted_suffixes(codes, lens):
    """(read, offset) of every suffix in sorted order: stable sorts by 31-base
    windows (A-padded, 62 bits) from the last to the first, starting from the
    order (suffix length, read)."""
    n, width = codes.shape
    cols = torch.arange(width + 1, device="cuda")
    length = lens[:, None] - cols[None, :]
    read, offset = (length >= 0).nonzero(as_tuple=True)
    order = torch.argsort(length[read, offset], stable=True)
    padded = torch.where(cols[None, :width] < lens[:, None], codes, torch.zeros_like(codes))
    window = torch.zeros((n, width + 1), dtype=torch.int64, device="cuda")
    for k in range(width - 1, -1, -1):
        window[:, k] = (window[:, k + 1] >> 2) + (padded[:, k].to(torch.int64) << 60)
    for c0 in range((width - 1) // 31 * 31, -1, -31):
        at = offset[order] + c0
        key = torch.where(at <= width, window[read[order], at.clamp(max=width)], torch.zeros_like(at))
        order = order[torch.argsort(key, stable=True)]
    return read[order], offset[order]


def _expected(codes, lens, with_sa=False):
    read, offset = _sorted_suffixes(codes, lens)
    whole = offset == 0
    symbol = torch.where(whole, 0, codes[read, (offset - 1).clamp(min=0)].to(torch.int64))
    dollar = torch.empty(codes.shape[0], dtype=torch.int64, device="cuda")
    dollar[read[whole]] = whole.nonzero().reshape(-1)
    counts = torch.bincount(torch.where(whole, 0, symbol + 1), minlength=5)
    out = (_packed(symbol.to(torch.uint8)), dollar, counts)
    return out + ((read << 16) | offset,) if with_sa else out


def exact(case, seed):
    kind = case["kind"]
    if kind in ("batch", "serve"):
        found = []
        for j, (n, length, genome) in enumerate(_specs(case)):
            codes = torch.cat(list(_blocks(n, length, genome, False, _generator(seed, j + 1))))
            found.append(_expected(codes, torch.full((n,), length, device="cuda")))
        return found
    if kind == "part" or case["reads"] * (case["length"] + 1) > 150_000_000:
        return None
    if kind == "mixed":
        flat, lens = _mixed_codes(case, seed)
        codes = torch.zeros((case["reads"], case["length"]), dtype=torch.uint8, device="cuda")
        codes[torch.arange(case["length"], device="cuda")[None, :] < lens[:, None]] = flat
        return _expected(codes, lens)
    codes = torch.cat(list(_blocks(case["reads"], case["length"], case["genome"], case.get("repeats", False), _generator(seed))))
    lens = torch.full((case["reads"],), case["length"], device="cuda")
    return _expected(codes, lens, kind == "sa")
