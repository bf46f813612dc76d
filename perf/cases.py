"""The work that a user of this package has it do, as cases that can be timed and compared.

Every case goes through the package's public entry points (paper_1807_09932_gb300.ebic). The sizes
are those of the package's own workloads (synth.config1 to config5: matrices of 1,000 to 436,444
rows and 20 to 500 columns, populations of 200 to 3,200 candidates of 2 to 64 columns), with the
paper's largest population (65,535) at the top. Five paths:

  score   one generation scored against the archive on a matrix with a pair table
          (ebic_eval_fitness: counts and fitness), as an EBIC search does each generation
  direct  one population scored on a matrix as loaded, without a pair table: counts and row
          bitmaps (ebic_eval_population), then fitness and overlaps (ebic_fitness)
  open    a data set opened: float32 values -> loaded matrix -> pair table -> the first
          population's counts and bitmaps
  batch   the generations of many runs on several matrices in one replay (ebic_batch_run), as
          the server and a study over several data sets do
  run     a whole EBIC search (ebic_run) with its archive as the result
"""
import numpy as np
import torch

from paper_1807_09932_gb300 import ebic

DEV = "cuda:0"


def listed():
    return [
        # the smallest data set (synth.config1's shape): a call is mostly launches and latency
        dict(name="score_small", path="score", rows=1000, cols=50, population=200, lmin=2,
             lmax=10, archive=20, nan=0.0, negative=False, exclude=True, beta=False),
        # an expression data set (synth.config2): 16-bit ranks, decreasing trends also count
        dict(name="score_expression", path="score", rows=20000, cols=200, population=1600,
             lmin=2, lmax=20, archive=20, nan=0.01, negative=True, exclude=True, beta=False),
        # a methylation data set (synth.config3), the headline workload of bench.py
        dict(name="score_methylation", path="score", rows=436444, cols=64, population=1600,
             lmin=2, lmax=16, archive=20, nan=0.005, negative=False, exclude=True, beta=True),
        # the same data set with the paper's largest population
        dict(name="score_largest", path="score", rows=436444, cols=64, population=65535, lmin=2,
             lmax=16, archive=20, nan=0.005, negative=False, exclude=True, beta=True),
        # a caller who scores a matrix as loaded and keeps bitmaps and overlaps: 8-bit ranks
        dict(name="direct_methylation", path="direct", rows=436444, cols=64, population=1600,
             lmin=2, lmax=16, archive=20, nan=0.005, negative=False, exclude=True, beta=True),
        # the same on the expression data set: 16-bit ranks, both trends
        dict(name="direct_expression", path="direct", rows=20000, cols=200, population=1600,
             lmin=2, lmax=20, archive=20, nan=0.01, negative=True, exclude=True, beta=False),
        # a wide data set of synth.config4's range, candidates up to the longest allowed, sizes
        # that no tile divides
        dict(name="direct_wide", path="direct", rows=50021, cols=457, population=1599, lmin=2,
             lmax=64, archive=20, nan=0.005, negative=False, exclude=True, beta=False),
        # opening the methylation data set: once per study, before any generation
        dict(name="open_methylation", path="open", rows=436444, cols=64, population=1600, lmin=2,
             lmax=6, archive=0, nan=0.005, negative=False, exclude=True, beta=True),
        # opening the wide data set
        dict(name="open_wide", path="open", rows=50021, cols=457, population=1600, lmin=2, lmax=6,
             archive=0, nan=0.005, negative=False, exclude=True, beta=False),
        # 64 populations on 8 matrices (synth.config4's range), each scored against its archive
        dict(name="batch_study", path="batch", matrices=8, rows=5000, rows_most=200000, cols=20,
             cols_most=500, requests=64, population=200, population_most=3200, lmin=2, lmax=64,
             archive=20, nan=0.005, negative=False, exclude=True, beta=False),
        # a short search on the expression data set with the default (host) generation loop
        dict(name="run_expression", path="run", rows=20000, cols=200, population=1600, lmin=2,
             lmax=6, archive=20, nan=0.01, negative=True, exclude=True, beta=False,
             generations=10, on_device=False),
        # a short search on the methylation data set with the generation loop on the device
        dict(name="run_methylation", path="run", rows=436444, cols=64, population=1600, lmin=2,
             lmax=6, archive=20, nan=0.005, negative=False, exclude=True, beta=True,
             generations=10, on_device=True),
    ]


def _log(rng, lo, hi):
    return int(round(lo * (hi / lo) ** rng.random()))


def draw(rng):
    """One case of the ranges above: rows, columns, populations and lengths over their whole
    ranges, both trend options, both missing-value options, archives of none to 64 members."""
    path = rng.choice(["score", "score", "score", "direct", "direct", "open", "batch", "run"])
    rows, cols = _log(rng, 1000, 436444), _log(rng, 8, 500)
    while path != "direct" and rows * cols * cols > 1.2e10:  # a pair table of at most 1.5 GB
        rows, cols = _log(rng, 1000, 436444), _log(rng, 8, 500)
    lmax = min(cols, rng.choice([6, 10, 16, 20, 64]))
    # the listed cases' largest work per path bounds a drawn population
    most = {"score": 2.2e11, "direct": 8e9, "open": 8e9}.get(path, 8e9)
    population = max(50, min(_log(rng, 50, 65535 if path == "score" else 6400),
                             int(most / rows / (lmax + 2) * 2)))
    c = dict(path=path, rows=rows, cols=cols, population=population, lmin=rng.choice([1, 2]),
             lmax=lmax, archive=rng.choice([0, 7, 20, 33, 64]), nan=rng.choice([0.0, 0.005, 0.05]),
             negative=rng.random() < 0.4, exclude=rng.random() < 0.8, beta=rng.random() < 0.5)
    if path == "batch":
        c.update(matrices=rng.randint(2, 8), rows=rng.randint(1000, 8000),
                 rows_most=_log(rng, 20000, 150000), cols=rng.randint(8, 40),
                 cols_most=rng.randint(60, 400), requests=rng.randint(4, 64),
                 population=rng.randint(50, 400), population_most=rng.randint(600, 3000), lmax=64)
    if path == "run":
        c.update(population=_log(rng, 100, 1600), archive=rng.choice([7, 20, 32]), lmin=2,
                 lmax=min(cols, 6), generations=rng.randint(3, 10), on_device=rng.random() < 0.5)
    return c


# ---- inputs ---------------------------------------------------------------------------------

def _matrix(gen, rows, cols, case):
    """float32 [rows, cols]: a normal or Beta(0.5, 0.5) background, planted row-disjoint trend
    biclusters (every third decreasing when decreasing trends count), uniformly missing values.
    Returns the values and the planted column orders."""
    x = torch.randn(rows, cols, generator=gen, device=DEV)
    if case["beta"]:
        x = torch.sin(0.5 * torch.pi * torch.rand(rows, cols, generator=gen, device=DEV)) ** 2
    perm = torch.randperm(rows, generator=gen, device=DEV)
    planted, per = [], max(1, rows // 16)
    for k in range(10):
        n = min(cols, 5 + (k * 7) % 12)
        order = torch.randperm(cols, generator=gen, device=DEV)[:n]
        at = perm[k * per:(k + 1) * per - (k * per) // 23]
        down = case["negative"] and k % 3 == 2
        x[at.unsqueeze(1), order.unsqueeze(0)] = x[at][:, order].sort(dim=1, descending=down)[0]
        planted.append(order.tolist())
    if case["nan"] > 0:
        x[torch.rand(rows, cols, generator=gen, device=DEV) < case["nan"]] = float("nan")
    return x.contiguous(), planted


def _lists(gen, n, cols, lmin, lmax):
    """n candidates of lmin to lmax distinct columns in random order, as CSR tensors (cols int16,
    offsets int32) on the device."""
    lmax = min(lmax, cols)
    lmin = min(lmin, lmax)
    lens = torch.randint(lmin, lmax + 1, (n,), generator=gen, device=DEV)
    picks = torch.rand(n, cols, generator=gen, device=DEV).argsort(dim=1)[:, :lmax]
    keep = torch.arange(lmax, device=DEV).unsqueeze(0) < lens.unsqueeze(1)
    offs = torch.zeros(n + 1, dtype=torch.int64, device=DEV)
    offs[1:] = lens.cumsum(0)
    return picks[keep].to(torch.int16), offs.to(torch.int32)


def _csr(lists):
    offs = [0]
    for c in lists:
        offs.append(offs[-1] + len(c))
    return (torch.tensor([v for c in lists for v in c] or [0], dtype=torch.int16, device=DEV),
            torch.tensor(offs, dtype=torch.int32, device=DEV))


def _archive(planted, k):
    """k column orders, as a search that has found the planted biclusters holds them: the planted
    orders, then parts of them."""
    out = []
    for i in range(k):
        p = planted[i % len(planted)]
        turn = i // len(planted)
        out.append(p if turn == 0 else p[turn % max(1, len(p) - 3):][:max(1, 3 + (i % 5))])
    return out


def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed) * 7919 + 13)
    return g


def _shapes(case):
    """batch: the matrices' (rows, cols) and the requests' (matrix, population), spread over the
    case's ranges whatever the seed."""
    n, r = case["matrices"], case["requests"]
    grow = case["rows_most"] / case["rows"]
    mats = [(int(round(case["rows"] * grow ** (i / max(1, n - 1)))),
             case["cols"] + (case["cols_most"] - case["cols"]) * ((i * 5) % n) // max(1, n - 1))
            for i in range(n)]
    reqs = [(i % n, case["population"] + (case["population_most"] - case["population"])
             * ((i * 29) % r) // max(1, r - 1)) for i in range(r)]
    return mats, reqs


def _population(gen, x, planted, case, n):
    cols, offs = _lists(gen, n, x.shape[1], case["lmin"], case["lmax"])
    arch = _archive(planted, case["archive"])
    return cols, offs, arch


class _Scored:
    """A matrix, a population, an archive and the output buffers of one request."""

    def __init__(self, m, cols, offs, arch, case, bitmaps=False):
        self.m, self.cols, self.offs, self.n = m, cols, offs, offs.numel() - 1
        self.flags = ebic.EBIC_NEGATIVE_TRENDS if case["negative"] else 0
        self.k = len(arch)
        self.acols, self.aoffs = _csr(arch)
        self.abm = torch.zeros(max(1, self.k), m.words, dtype=torch.int32, device=DEV)
        if self.k:
            counts = torch.empty(self.k, dtype=torch.int32, device=DEV)
            ebic.eval_population(m, self.acols, self.aoffs, negative=case["negative"],
                                 counts=counts, bitmaps=self.abm)
        self.counts = torch.zeros(self.n, dtype=torch.int32, device=DEV)
        self.fitness = torch.zeros(self.n, dtype=torch.int64, device=DEV)
        self.bitmaps = torch.zeros(self.n, m.words, dtype=torch.int32, device=DEV) if bitmaps else None
        self.overlaps = torch.zeros(self.n, max(1, self.k), dtype=torch.int32, device=DEV) if bitmaps else None


class _Batch:
    """A batch handle, freed with the state."""

    def __init__(self, n):
        self.handle = ebic.ebic_batch_create(n)

    def __del__(self):
        ebic.ebic_batch_free(self.handle)


def prepare(case, seed):
    gen, path = _gen(seed), case["path"]
    if path == "batch":
        mats, reqs = _shapes(case)
        ms, plants = [], []
        for r, c in mats:
            x, planted = _matrix(gen, r, c, case)
            ms.append(ebic.Matrix(x, exclude_missing=case["exclude"]))
            ms[-1].build_pairs()
            plants.append(planted)
        scored = []
        for i, n in reqs:
            cols, offs = _lists(gen, n, mats[i][1], case["lmin"], case["lmax"])
            scored.append(_Scored(ms[i], cols, offs, _archive(plants[i], case["archive"]), case))
        items = [(q.m.handle, q.cols, q.offs, q.n, q.flags, q.counts, None, q.acols, q.aoffs,
                  q.abm, q.k, q.fitness) for q in scored]
        return dict(path=path, scored=scored, batch=_Batch(len(items)), n=len(items),
                    requests=ebic.make_requests(items))
    x, planted = _matrix(gen, case["rows"], case["cols"], case)
    cols, offs, arch = _population(gen, x, planted, case, case["population"])
    if path == "open":
        n, words = offs.numel() - 1, ebic.words(case["rows"])
        return dict(path=path, x=x, exclude=case["exclude"], negative=case["negative"], cols=cols,
                    offs=offs, counts=torch.zeros(n, dtype=torch.int32, device=DEV),
                    bitmaps=torch.zeros(n, words, dtype=torch.int32, device=DEV))
    m = ebic.Matrix(x, exclude_missing=case["exclude"])
    if path != "direct":
        m.build_pairs()
    if path == "run":
        p = ebic.ebic_params_default(
            population=case["population"], generations=case["generations"],
            archive_size=case["archive"], max_init_len=case["lmax"], max_len=min(64, case["cols"]),
            flags=(ebic.EBIC_NEGATIVE_TRENDS if case["negative"] else 0)
            | (ebic.EBIC_RUN_ON_DEVICE if case["on_device"] else 0), seed=int(seed) + 1)
        return dict(path=path, m=m, params=p)
    return dict(path=path, q=_Scored(m, cols, offs, arch, case, bitmaps=path == "direct"))


def run(state):
    path = state["path"]
    if path == "score":
        q = state["q"]
        rc = ebic.ebic_eval_fitness(q.m.handle, q.cols, q.offs, q.n, q.flags, q.acols, q.aoffs,
                                    q.abm, q.k, q.counts, None, q.fitness, None)
        if rc:
            raise ebic.EbicError(rc, "ebic_eval_fitness")
        return dict(counts=q.counts, fitness=q.fitness)
    if path == "direct":
        q = state["q"]
        rc = ebic.ebic_eval_population(q.m.handle, q.cols, q.offs, q.n, q.flags, q.counts,
                                       q.bitmaps)
        if not rc:
            rc = ebic.ebic_fitness(q.m.handle, q.cols, q.offs, q.n, q.counts, q.bitmaps, q.acols,
                                   q.aoffs, q.abm, q.k, 0, q.fitness, q.overlaps)
        if rc:
            raise ebic.EbicError(rc, "ebic_eval_population, ebic_fitness")
        return dict(counts=q.counts, bitmaps=q.bitmaps, fitness=q.fitness, overlaps=q.overlaps)
    if path == "open":
        with ebic.Matrix(state["x"], exclude_missing=state["exclude"]) as m:
            m.build_pairs()
            ebic.eval_population(m, state["cols"], state["offs"], negative=state["negative"],
                                 counts=state["counts"], bitmaps=state["bitmaps"])
        return dict(counts=state["counts"], bitmaps=state["bitmaps"])
    if path == "batch":
        rc = ebic.ebic_batch_run(state["batch"].handle, state["requests"], state["n"])
        if rc:
            raise ebic.EbicError(rc, "ebic_batch_run")
        # one tensor of all requests' counts and one of all their fitness
        return dict(counts=torch.cat([q.counts for q in state["scored"]]),
                    fitness=torch.cat([q.fitness for q in state["scored"]]))
    r = ebic.ebic_run(state["m"].handle, state["params"])
    # the archive in arrays of one size, whatever number of members it holds (the rest zero)
    k, n = state["params"].archive_size, len(r["counts"])
    out = dict(cols=np.zeros(k * 64, np.int32), offsets=np.zeros(k + 1, np.int64),
               counts=np.zeros(k, np.int64), quality=np.zeros(k, np.int64),
               bitmaps=np.zeros((k, r["bitmaps"].shape[1]), np.uint32))
    out["cols"][:len(r["cols"])] = r["cols"]
    out["offsets"][:n + 1] = r["offsets"]
    for name in ("counts", "quality", "bitmaps"):
        out[name][:n] = r[name]
    return out


def work(case):
    """One pass's bytes (the ranks of the matrix and the lists read once, the results written
    once) and operations (a comparison per row and consecutive pair of a candidate's columns; an
    AND with popcount per 32 rows, candidate and archive member). A search counts its scoring."""
    def scoring(rows, cols, n, case, bitmaps):
        words, lens = (rows + 31) // 32, (min(case["lmin"], cols) + min(case["lmax"], cols)) / 2
        k, both = case["archive"], 2 if case["negative"] else 1
        b = rows * cols * (1 if cols <= 127 else 2) + n * (2 * lens + 4) + k * words * 4 + n * 12
        if bitmaps:
            b += n * words * 4 + n * k * 4
        return b, n * rows * max(1.0, lens - 1) * both + n * k * words

    path = case["path"]
    if path == "batch":
        mats, reqs = _shapes(case)
        every = [scoring(*mats[i], n, case, False) for i, n in reqs]
        # a matrix is read once, whatever number of requests it has
        again = sum(mats[i][0] * mats[i][1] * (1 if mats[i][1] <= 127 else 2)
                    for j, (i, n) in enumerate(reqs) if j >= len(mats))
        return dict(bytes=sum(b for b, _ in every) - again, flops=sum(f for _, f in every))
    rows, cols = case["rows"], case["cols"]
    b, f = scoring(rows, cols, case["population"], case, path in ("direct", "open"))
    if path == "open":  # the values read, the pair table written
        b += rows * cols * 4 + cols * cols * ((rows + 31) // 32) * 4
        f += cols * cols * rows
    if path == "run":
        b, f = b * case["generations"], f * case["generations"]
    return dict(bytes=b, flops=f)


def exact(case, seed):
    """The counts, bitmaps, fitness and overlaps by plain comparisons of the 64-bit values, a
    candidate at a time; None for a batch, a search and the largest populations."""
    if case["path"] not in ("score", "direct", "open"):
        return None
    if case["population"] * (case["lmin"] + case["lmax"]) > 150000:
        return None
    gen = _gen(seed)
    x, planted = _matrix(gen, case["rows"], case["cols"], case)
    cols, offs, arch = _population(gen, x, planted, case, case["population"])
    cols, offs = cols.tolist(), offs.tolist()
    if not case["exclude"]:
        x = torch.nan_to_num(x, nan=0.0, posinf=float("inf"), neginf=float("-inf"))
    v = x.t().contiguous().double()
    here = ~torch.isnan(v)
    rows, words = case["rows"], (case["rows"] + 31) // 32

    def follows(c):
        up = here[c[0]].clone()
        for a in c[1:]:
            up &= here[a]
        down = up.clone()
        for a, b in zip(c, c[1:]):
            up &= v[a] <= v[b]
            if case["negative"]:
                down &= v[a] >= v[b]
        return up | down if case["negative"] else up

    def packed(mask):
        bits = torch.zeros(words * 32, dtype=torch.int64, device=DEV)
        bits[:rows] = mask
        w = (bits.view(words, 32) << torch.arange(32, device=DEV)).sum(1)
        return torch.where(w >= 2 ** 31, w - 2 ** 32, w).to(torch.int32)

    k = len(arch)
    amask = torch.stack([follows(a) for a in arch]) if k else None
    acount = amask.sum(1).tolist() if k else []
    bitmaps = case["path"] != "score"
    counts, fits, overs, maps = [], [], [], []
    for i in range(len(offs) - 1):
        c = cols[offs[i]:offs[i + 1]]
        mask = follows(c)
        shift = min(len(c), 33) - 1
        n = mask.sum()
        over = (amask & mask).sum(1) if k else None
        got = [n] + ([over] if k else [])
        got = torch.cat([t.reshape(-1) for t in got]).tolist()
        worst = 0
        for j, a in enumerate(arch):
            if set(a) & set(c) and acount[j] << (min(len(a), 33) - 1) >= got[0] << shift:
                worst = max(worst, got[1 + j])
        counts.append(got[0])
        fits.append((got[0] - worst) << shift)
        overs.append(got[1:] or [0])
        if bitmaps:
            maps.append(packed(mask))
    out = dict(counts=torch.tensor(counts, dtype=torch.int32))
    if case["path"] != "open":
        out["fitness"] = torch.tensor(fits, dtype=torch.int64)
    if bitmaps:
        out["bitmaps"] = torch.stack(maps)
    if case["path"] == "direct":
        out["overlaps"] = torch.tensor(overs, dtype=torch.int32)
    return out
