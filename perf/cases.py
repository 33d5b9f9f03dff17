"""Performance cases of the library: what its users have it do, and the inputs for it.

A case is a plain dict; `kind` says which public entry points it goes through:

  search      serve.search: a pass of query regions (host bytes) against a resident index
  serve       DeviceServer: a wave of query regions through the continuous-batching server
  selfsearch  Context.selfsearch: stage by stage, every intermediate returned
  onecall     Context.sedef_selfsearch: the whole self-search of a device sequence in one call
  host        Context.sedef_selfsearch_host: the same from host bytes to host candidates
  graph       Graph.launch / wait: the captured self-search pass
  index       sedef_pack, sedef_sketch, sedef_index: what makes a genome searchable
  regions     sedef_qgram, sedef_extend, sedef_chain2: from kept seeds to final duplications

The genomes have the shapes of the repository's own workloads (synth.py): random bases, soft-masked
repeat families of 300 and 6,000 bases at 80-95% identity, planted duplications of log-uniform
length in both orientations with substitutions and small indels, runs of N in assemblies.  They are
drawn on the GPU here, so that gigabase inputs take about a second.  Every output is whole numbers,
so there is no rounding for an exact() to measure.
"""
import ctypes
import math

import numpy as np
import torch

from paper_1807_00205_gb300 import binding, serve

ACGT = (65, 67, 71, 84)
# The 24 sequences of the human-scale assembly and the 200 genomes of the batch are
# drawn from these lengths.
ASSEMBLY_LO, ASSEMBLY_HI = 50_000_000, 250_000_000


def listed():
    return [
        # one short region asked of a resident human-scale index: the smallest request a
        # server sees, all latency
        {"name": "search-10k", "kind": "search", "target": 3_100_000_000, "nseq": 24,
         "requests": 1, "req_lo": 10_007, "req_hi": 10_007},
        # one request of the serving workload's mean length against the same index
        {"name": "search-1m", "kind": "search", "target": 3_100_000_000, "nseq": 24,
         "requests": 1, "req_lo": 950_000, "req_hi": 950_000},
        # a pass of requests of the serving workload's uneven lengths (10 kbp to 5 Mbp)
        {"name": "search-24", "kind": "search", "target": 3_100_000_000, "nseq": 24,
         "requests": 24, "req_lo": 10_000, "req_hi": 5_000_000},
        # the same requests through the continuous-batching server, a gigabase index
        {"name": "serve-16", "kind": "serve", "target": 1_000_000_000, "nseq": 8,
         "requests": 16, "req_lo": 10_000, "req_hi": 2_000_000},
        # the small uppercase genome, stage by stage with every intermediate kept
        {"name": "plain-2m", "kind": "selfsearch", "genomes": 1, "lo": 2_000_000,
         "hi": 2_000_000, "gc": 0.5, "mask": 0.0, "sds_lo": 20, "sds_hi": 20, "sd_len": 20_000,
         "mode": 1},
        # one chromosome: repeats, gaps, many duplications
        {"name": "chromosome-100m", "kind": "onecall", "genomes": 1, "lo": 100_000_000,
         "hi": 100_000_000, "gc": 0.41, "mask": 0.4, "sds_lo": 2000, "sds_hi": 2000,
         "sd_len": 200_000, "gaps": True, "mode": 1},
        # a small assembly of several sequences searched against itself: longer posting
        # lists, duplications between sequences
        {"name": "assembly-240m", "kind": "onecall", "genomes": 6, "lo": 20_000_000,
         "hi": 80_000_000, "total": 240_000_011, "gc": 0.41, "mask": 0.5, "sds_lo": 300,
         "sds_hi": 300, "sd_len": 200_000, "inter": 0.3, "gaps": True, "mode": 1},
        # the batch: 200 independent genomes of uneven size in one pass
        {"name": "batch-200", "kind": "onecall", "genomes": 200, "lo": 1_000_000,
         "hi": 20_000_000, "gc": 0.41, "mask": 0.3, "sds_lo": 50, "sds_hi": 500,
         "sd_len": 50_000, "mode": 2},
        # a smaller batch end to end from page-locked host memory
        {"name": "host-40", "kind": "host", "genomes": 40, "lo": 1_000_000, "hi": 20_000_000,
         "gc": 0.41, "mask": 0.3, "sds_lo": 50, "sds_hi": 500, "sd_len": 50_000, "mode": 2},
        # a captured pass over a few genomes, replayed
        {"name": "graph-12", "kind": "graph", "genomes": 12, "lo": 700_000, "hi": 4_000_000,
         "gc": 0.41, "mask": 0.3, "sds_lo": 20, "sds_hi": 60, "sd_len": 20_000, "mode": 2},
        # a human-scale assembly made searchable
        {"name": "index-3100m", "kind": "index", "target": 3_100_000_000, "nseq": 24},
        # the steps after the seeds of a small genome
        {"name": "regions-4m", "kind": "regions", "genomes": 1, "lo": 4_000_000,
         "hi": 4_000_000, "gc": 0.41, "mask": 0.3, "sds_lo": 30, "sds_hi": 30, "sd_len": 20_000,
         "mode": 1},
    ]


def _log(rng, lo, hi):
    return int(math.exp(rng.uniform(math.log(lo), math.log(hi))))


def draw(rng):
    kind = rng.choice(["search", "search", "serve", "selfsearch", "onecall", "onecall", "host",
                       "graph", "index", "regions"])
    if kind in ("search", "serve"):
        n = rng.choice([1, 1, 2, 5, 12]) if kind == "search" else rng.randint(2, 16)
        lo = _log(rng, 10_000, 200_000)
        target = _log(rng, 100_000_000, 3_100_000_000 if kind == "search" else 1_000_000_000)
        return {"kind": kind, "target": target, "nseq": rng.randint(1, max(1, min(24, target // 60_000_000))),
                "requests": n, "req_lo": lo, "req_hi": _log(rng, 2 * lo, 2_000_000)}
    if kind == "index":
        n = _log(rng, 1_000_000, 3_000_000_000)
        return {"kind": kind, "target": n, "nseq": rng.randint(1, max(1, min(24, n // 60_000_000))),
                "k": rng.choice([12, 12, 11, 13, 14]), "w": rng.choice([16, 16, 10, 24, 50])}
    c = {"kind": kind, "gc": round(rng.uniform(0.38, 0.5), 3), "mask": round(rng.uniform(0.0, 0.5), 3)}
    mode = rng.choice([1, 2]) if kind in ("onecall", "host", "selfsearch") else 2
    if kind == "regions":
        mode = 1
    if mode == 1:  # one genome
        top = {"onecall": 100_000_000, "host": 60_000_000, "selfsearch": 30_000_000,
               "regions": 6_000_000}[kind]
        n = _log(rng, 1_000_000, top)
        c.update(genomes=1, lo=n, hi=n, sds_lo=10, sds_hi=max(11, n // 100_000),
                 sd_len=rng.randint(5_000, 50_000), gaps=n > 20_000_000)
    else:  # a batch
        c.update(genomes=rng.randint(2, 12 if kind == "graph" else 40), lo=rng.randint(300_000, 1_000_000),
                 hi=_log(rng, 2_000_000, 4_000_000 if kind == "graph" else 20_000_000), sds_lo=10,
                 sds_hi=rng.randint(11, 60 if kind == "graph" else 300), sd_len=rng.randint(5_000, 50_000))
    c["mode"] = mode
    if kind in ("onecall", "host", "selfsearch"):
        c["w"] = rng.choice([16, 16, 16, 12, 24])
        c["step"] = rng.choice([250, 250, 125, 400])
        if mode == 2:
            c["k"] = rng.choice([12, 12, 12, 11, 13])
        if rng.random() < 0.2:
            c["max_occ"] = rng.choice([200, 1000])
    return c


# ------------------------------------------------------------- the inputs --

class _Maker:
    """Genomes drawn on the GPU from one seed.  Every write goes to places that no other write of
    the same operation has, so the same seed gives the same bytes."""

    def __init__(self, seed):
        self.rng = np.random.default_rng(seed)
        self.gen = torch.Generator(device="cuda")
        self.gen.manual_seed(seed)
        self.acgt = torch.tensor(ACGT, dtype=torch.uint8, device="cuda")
        code = torch.zeros(256, dtype=torch.uint8)
        comp = torch.arange(256, dtype=torch.uint8)
        for x, (a, b) in enumerate(zip(b"ACGT", b"TGCA")):
            code[a] = code[a + 32] = x
            comp[a], comp[a + 32] = b, b + 32
        self.code, self.comp = code.cuda(), comp.cuda()

    def uniform(self, *shape):
        return torch.rand(*shape, generator=self.gen, device="cuda")

    def bases(self, n, gc):
        out = torch.empty(n, dtype=torch.uint8, device="cuda")
        at = (1.0 - gc) / 2.0
        for a in range(0, n, 1 << 27):
            u = self.uniform(min(1 << 27, n - a))
            x = (u >= at).to(torch.uint8) + (u >= 0.5).to(torch.uint8) + (u >= 1.0 - at).to(torch.uint8)
            out[a:a + len(u)] = self.acgt[x.int()]
        return out

    def repeats(self, seq, frac, gc):
        """Soft-masked copies of a 6,000- and a 300-base consensus over about `frac` of seq."""
        if frac <= 0:
            return
        each = 1.0 - math.sqrt(1.0 - frac)
        for flen in (6000, 300):
            n = int(each * len(seq) / flen)
            if n < 1:
                continue
            cons = self.code[self.bases(flen, gc).int()]
            room = len(seq) // n  # a copy has a stretch of its own
            start = torch.arange(n, device="cuda") * room + (self.uniform(n) * (room - flen)).long()
            ident = 0.80 + 0.15 * self.uniform(n, 1)
            step = max(1, (1 << 26) // flen)
            for a in range(0, n, step):
                b = min(n, a + step)
                u = self.uniform(b - a, flen)
                sub = u >= ident[a:b]
                shift = 1 + (self.uniform(b - a, flen) * 3).to(torch.uint8).clamp_(max=2)
                row = (cons + shift * sub) & 3
                at = start[a:b, None] + torch.arange(flen, device="cuda")
                seq[at] = self.acgt[row.int()] | 32

    def copies(self, seq, src, length, ident, rc):
        """Mutated copies of seq[src, src + length), one after another: (bases, lengths)."""
        n, total = len(src), int(length.sum())
        L = torch.from_numpy(length).cuda()
        sd = torch.repeat_interleave(torch.arange(n, device="cuda"), L)
        begin = torch.cumsum(L, 0) - L
        at = torch.from_numpy(src).cuda()[sd] + torch.arange(total, device="cuda") - begin[sd]
        base = seq[at]
        ev = self.uniform(total) < (1.0 - torch.from_numpy(ident).float().cuda())[sd]
        what = self.uniform(total)
        size = 1 + (self.uniform(total) * 5).long().clamp_(max=4)
        sub = ev & (what < 0.8)
        new = (self.code[base.int()] + 1 + (self.uniform(total) * 3).to(torch.uint8).clamp_(max=2)) & 3
        base = torch.where(sub, self.acgt[new.int()] | (base & 32), base)
        ins = torch.where(ev & (what >= 0.8) & (what < 0.9), size, 0)
        gone = torch.zeros(total + 8, dtype=torch.int32, device="cuda")
        dp = torch.nonzero(ev & (what >= 0.9))[:, 0]
        one = torch.ones(len(dp), dtype=torch.int32, device="cuda")
        gone.index_add_(0, dp, one)
        gone.index_add_(0, dp + size[dp], -one)
        count = ins + (torch.cumsum(gone, 0)[:total] <= 0)
        pick = torch.repeat_interleave(torch.arange(total, device="cuda"), count)
        rank = torch.arange(len(pick), device="cuda") - (torch.cumsum(count, 0) - count)[pick]
        out = base[pick]
        rand = self.acgt[(self.uniform(len(pick)) * 4).int().clamp_(max=3)] | (out & 32)
        out = torch.where(rank < ins[pick], rand, out)
        osd = sd[pick]
        olen = torch.zeros(n, dtype=torch.int64, device="cuda").index_add_(0, sd, count)
        obeg = torch.cumsum(olen, 0) - olen
        r = torch.arange(len(out), device="cuda") - obeg[osd]
        flip = torch.from_numpy(rc).cuda()[osd]
        out = torch.where(flip, self.comp[out.int()], out)
        place = torch.empty_like(out)
        place[obeg[osd] + torch.where(flip, olen[osd] - 1 - r, r)] = out
        return place, olen

    def plant(self, seq, offsets, counts, len_hi, id_lo, id_hi, inter=0.0):
        """counts[s] duplications of 1,000..len_hi bases in sequence s.  They are written in
        layers whose places do not overlap; a later layer may copy an earlier one."""
        layers = {}
        size = np.diff(offsets)
        for s, c in enumerate(counts):
            top = min(len_hi, int(size[s]) // 8)
            if top <= 1000 or c < 1:
                continue
            L = np.exp(self.rng.uniform(math.log(1000), math.log(top), size=c)).astype(np.int64)
            room = L + L // 8 + 64
            layer = np.cumsum(room) // (int(size[s]) // 2)
            for y in np.unique(layer):
                m = layer == y
                slack = int(size[s]) - int(room[m].sum())
                if slack <= 0:
                    continue
                k = int(m.sum())
                dst = offsets[s] + np.cumsum(room[m]) - room[m] + \
                    np.sort((self.rng.random(k) * slack).astype(np.int64))
                other = np.where(self.rng.random(k) < inter, self.rng.integers(0, len(size), k), s)
                other = np.where(size[other] > 2 * L[m], other, s)
                src = offsets[other] + (self.rng.random(k) * (size[other] - L[m])).astype(np.int64)
                layers.setdefault(int(y), []).append((src, L[m], dst, room[m]))
        for y in sorted(layers):
            src, L, dst, room = (np.concatenate(v) for v in zip(*layers[y]))
            ident = self.rng.uniform(id_lo, id_hi, size=len(L))
            rc = self.rng.random(len(L)) < 0.5
            cut = np.concatenate([[0], np.flatnonzero(np.diff(np.cumsum(L) // (1 << 25))) + 1, [len(L)]])
            for a, b in zip(cut[:-1], cut[1:]):
                out, olen = self.copies(seq, src[a:b], L[a:b], ident[a:b], rc[a:b])
                sd = torch.repeat_interleave(torch.arange(int(b - a), device="cuda"), olen)
                r = torch.arange(len(out), device="cuda") - (torch.cumsum(olen, 0) - olen)[sd]
                ok = r < torch.from_numpy(room[a:b]).cuda()[sd]
                seq[(torch.from_numpy(dst[a:b]).cuda()[sd] + r)[ok]] = out[ok]

    def gaps(self, seq):
        for a in range(0, len(seq), 10_000_000):
            g = int(self.rng.integers(10_000, 50_001))
            room = min(10_000_000, len(seq) - a) - g
            if room > 0:
                a += int(self.rng.integers(0, room))
                seq[a:a + g] = ord("N")

    def genomes(self, case):
        """(device bytes, offsets) of a self-search case."""
        n = case["genomes"]
        lo, hi = case["lo"], case["hi"]
        size = np.exp(self.rng.uniform(math.log(lo), math.log(hi), size=n)).astype(np.int64) if hi > lo \
            else np.full(n, lo, dtype=np.int64)
        if case.get("total"):
            size = np.maximum(1_000_000, (size * (case["total"] / size.sum())).astype(np.int64))
        offsets = np.concatenate([[0], np.cumsum(size)]).astype(np.int64)
        seq = self.bases(int(offsets[-1]), case["gc"])
        for s in range(n):
            self.repeats(seq[int(offsets[s]):int(offsets[s + 1])], case["mask"], case["gc"])
        counts = self.rng.integers(case["sds_lo"], case["sds_hi"] + 1, size=n)
        self.plant(seq, offsets, counts, case["sd_len"], 0.75, 0.99, case.get("inter", 0.0))
        if case.get("gaps"):
            for s in range(n):
                self.gaps(seq[int(offsets[s]):int(offsets[s + 1])])
        return seq, offsets

    def assembly(self, total, nseq):
        """(device bytes, offsets) of an assembly of nseq chromosomes."""
        share = self.rng.uniform(ASSEMBLY_LO, ASSEMBLY_HI, size=nseq)
        offsets = np.concatenate([[0], np.cumsum(share / share.sum() * total)]).astype(np.int64)
        offsets[-1] = total
        seq = self.bases(total, 0.41)
        parts = [seq[int(offsets[s]):int(offsets[s + 1])] for s in range(nseq)]
        for x in parts:
            self.repeats(x, 0.5, 0.41)
        counts = np.diff(offsets) * 20_000 // 3_100_000_000  # 20,000 in 3.1 Gbp
        self.plant(seq, offsets, counts, 300_000, 0.75, 0.995, 0.3)
        for x in parts:
            self.gaps(x)
        return seq, offsets

    def regions(self, seq, offsets, case):
        """Query regions cut from the assembly, with 0-25% added mutation (host bytes)."""
        size = np.diff(offsets)
        out = []
        for _ in range(case["requests"]):
            n = int(math.exp(self.rng.uniform(math.log(case["req_lo"]), math.log(case["req_hi"] + 1))))
            s = int(self.rng.choice(len(size), p=size / size.sum()))
            n = min(n, int(size[s]))
            a = np.array([offsets[s] + int(self.rng.integers(0, size[s] - n + 1))])
            q, _ = self.copies(seq, a, np.array([n]), 1.0 - self.rng.uniform(0.0, 0.25, size=1),
                               self.rng.random(1) < 0.5)
            out.append(q.cpu().numpy())
        return out


_ctx = None


def _context():
    """The one context that a program keeps."""
    global _ctx
    if _ctx is None:
        _ctx = binding.Context(0)
    return _ctx


def _params(case, mode):
    return binding.params(self_mode=mode, **{k: case[k] for k in ("k", "w", "step", "max_occ") if k in case})


# The sizes of most outputs depend on the data.  A program keeps buffers that hold the largest it
# expects; a pass fills their first rows and gives the counts beside them.

def _bases(case):
    """An upper bound of a genome case's length, from the case alone."""
    if case["kind"] in ("index", "search", "serve"):
        return case["target"]
    return (case.get("total") or case["genomes"] * case["hi"]) + 1_000_000


def _device(n, dtype=torch.uint8):
    return torch.zeros(int(n), dtype=dtype, device="cuda")


def _put(buf, x):
    """x into the first rows of a buffer."""
    if len(x) > len(buf):
        raise ValueError("an output of %d is longer than the buffer of %d kept for it" % (len(x), len(buf)))
    buf[:len(x)] = x
    return buf


def prepare(case, seed):
    make = _Maker(seed)
    kind = case["kind"]
    ctx = _context()
    if kind in ("search", "serve"):
        p = binding.params(self_mode=0)
        seq, off = make.assembly(case["target"], case["nseq"])
        reqs = make.regions(seq, off, case)
        # the resident index, as serve.ResidentIndex builds it
        p1 = binding.params(self_mode=1)
        rec = ctx.sedef_sketch(*ctx.sedef_pack(seq), off, p1).clone()
        srt, tab = ctx.sedef_index(rec, p1)
        st = {"kind": kind, "ctx": ctx, "reqs": reqs, "p": p,
              "cands": [np.zeros((case["req_hi"] // 16 + 1024, 10), dtype=np.int32) for _ in reqs]}
        if kind == "search":
            st["index"] = serve.ResidentIndex.from_arrays(rec, srt, tab, off, p1)
        else:
            st["server"] = binding.DeviceServer(ctx, rec, srt, tab, off, p, slots=len(reqs),
                                                slot_bases=max(len(q) for q in reqs) + 1,
                                                idle_timeout_s=0.002)
        return st
    n = _bases(case)
    if kind == "index":
        seq, off = make.assembly(case["target"], case["nseq"])
        cap = n // 4 + 1024
        return {"kind": kind, "ctx": ctx, "seq": seq, "off": off, "p": _params(case, 1),
                "rec": _device(cap, torch.int64), "sorted": _device(cap, torch.int64),
                "off_table": _device(4 ** case.get("k", 12) + 1, torch.int32)}
    p = _params(case, case["mode"])
    seq, off = make.genomes(case)
    st = {"kind": kind, "ctx": ctx, "seq": seq, "off": off, "p": p,
          "cands": _device((n // 32 + 4096) * binding.CAND_DTYPE.itemsize)}
    if kind in ("selfsearch", "graph"):
        st.update(rec=_device(n // 4, torch.int64), runs=_device(n // 16 * binding.RUN_DTYPE.itemsize),
                  chains=_device(n // 32 * binding.CHAIN_DTYPE.itemsize))
    if kind == "selfsearch":
        st.update(sorted=_device(n // 4, torch.int64), packed=_device(n // 16, torch.int32),
                  mask=_device(n // 32, torch.int32), nbits=_device(n // 32, torch.int32))
    elif kind == "host":
        st["seq"] = seq.cpu().pin_memory().numpy()
        st["cands"] = np.zeros((n // 32 + 4096, 10), dtype=np.int32)
    elif kind == "graph":
        st["graph"] = ctx.selfsearch_graph(seq, off, p)
    elif kind == "regions":
        out = ctx.selfsearch(seq, off, p)
        p0 = binding.params_from_struct(p, min_unmasked=0)
        ext = ctx.sedef_sketch(out["packed"], out["mask"], out["nbits"], off, p0)
        st.update(ext=ext, **{k: out[k] for k in ("packed", "nbits", "runs", "nruns")})
        st.update(shared=_device(n // 16, torch.int32), ok=_device(n // 16),
                  regions=_device(n // 16 * binding.REGION_DTYPE.itemsize),
                  sds=_device(n // 16 * binding.SD_DTYPE.itemsize))
    return st


def _rows(cands):
    return np.ascontiguousarray(cands).view(np.int32).reshape(-1, 10)


def run(st):
    kind, ctx, p = st["kind"], st["ctx"], st["p"]
    if kind == "search":
        reqs = [serve.Request(rid=k, seq=q) for k, q in enumerate(st["reqs"])]
        serve.search(ctx, st["index"], reqs, p)
        return [len(r.cands) for r in reqs], [_put(b, _rows(r.cands)) for b, r in zip(st["cands"], reqs)]
    if kind == "serve":
        srv, slot_of, out = st["server"], {}, {}
        for k, q in enumerate(st["reqs"]):
            slot_of[srv.submit(q)] = k
        while len(out) < len(st["reqs"]):
            slot = srv.poll(0.01)
            if slot is not None:
                out[slot_of[slot]] = srv.finish(slot)
        return [len(out[k]) for k in range(len(out))], \
            [_put(b, _rows(out[k])) for k, b in enumerate(st["cands"])]
    if kind in ("selfsearch", "graph"):
        if kind == "selfsearch":
            out = ctx.selfsearch(st["seq"], st["off"], p)
        else:
            st["graph"].launch()
            st["graph"].wait()
            out = st["graph"].outputs()
        names = ("packed", "mask", "nbits", "rec", "sorted", "runs", "chains", "cands")
        return out["nruns"], out["nchains"], out["ncands"], {x: _put(st[x], out[x]) for x in names if x in st}, \
            out["off"]
    if kind == "onecall":
        cands, count = ctx.sedef_selfsearch(st["seq"], st["off"], p)
        return count, _put(st["cands"], cands)
    if kind == "host":
        cands = ctx.sedef_selfsearch_host(st["seq"], st["off"], p)
        return len(cands), _put(st["cands"], _rows(cands))
    if kind == "index":
        # the C entry points, into buffers that the program owns
        packed, mask, nbits = ctx.sedef_pack(st["seq"])
        off, count = np.ascontiguousarray(st["off"], dtype=np.int64), ctypes.c_int64()
        rec, srt, tab = st["rec"], st["sorted"], st["off_table"]
        status = ctx.lib.sedef_sketch(ctx.handle, packed.data_ptr(), mask.data_ptr(), nbits.data_ptr(),
                                      off.ctypes.data, len(off) - 1, ctypes.byref(p), rec.data_ptr(),
                                      len(rec), ctypes.byref(count))
        if status == 0:
            status = ctx.lib.sedef_index(ctx.handle, rec.data_ptr(), count.value, ctypes.byref(p),
                                         srt.data_ptr(), tab.data_ptr())
        if status != 0:
            raise binding.SedefError(status, ctx.lib.sedef_last_error().decode())
        return count.value, packed, mask, nbits, rec, srt, tab
    n = int(st["off"][-1])
    shared, ok, npass = ctx.sedef_qgram(st["packed"], st["nbits"], n, st["runs"], st["nruns"], p)
    regions, nregions = ctx.sedef_extend(st["runs"], st["nruns"], st["ext"], st["off"], st["ext"],
                                         st["off"], p, max_len=100_000)
    sds, nsds = ctx.sedef_chain2(st["packed"], st["nbits"], n, regions, nregions, p)
    return npass, nregions, nsds, _put(st["shared"], shared), _put(st["ok"], ok), \
        _put(st["regions"], regions), _put(st["sds"], sds)


def work(case):
    """Bytes that a pass cannot do without: each input read once, each output written once.  The
    operations are integer, not floating."""
    kind, w, k = case["kind"], case.get("w", 16), case.get("k", 12)
    if kind in ("search", "serve"):
        lo, hi = case["req_lo"], case["req_hi"]
        q = case["requests"] * ((hi - lo) / math.log(hi / lo) if hi > lo else lo)
        recs = q * 2 / (w + 1)
        index = case["target"] * 2 / (w + 1) * 0.5  # half of it masked repeats
        # the postings of the queries' distinct hashes (of 4^k / 2 canonical ones)
        nhash = 4 ** k / 2
        return {"bytes": q + 8 * index * (1 - math.exp(-recs / nhash)), "flops": 0}
    if kind == "index":
        n = case["target"]
        return {"bytes": n + n / 2 + 2 * 8 * n * 1.2 / (w + 1) + 4 * 4 ** k, "flops": 0}
    lo, hi = case["lo"], case["hi"]
    n = case.get("total") or case["genomes"] * ((hi - lo) / math.log(hi / lo) if hi > lo else lo)
    if kind == "selfsearch":  # with the packed words, both record arrays and the offsets
        return {"bytes": n + n / 2 + 2 * 8 * n * 2 / (w + 1) + 4 * 4 ** k, "flops": 0}
    if kind == "regions":  # packed words, N bits and the extension sketch
        return {"bytes": n * 3 / 8 + 8 * n * 2 / (w + 1), "flops": 0}
    return {"bytes": n + n / 160, "flops": 0}
