"""What the phasing path is measured on: whole passes as a phasing program runs them
(fragments -> graph build -> bSB solve -> haplotypes), over the sizes, precisions, graph
kinds and options in use, and the BF16 product entry point on its own.

Sizes come from the package's generators (synth.py), the benchmark's workloads and the
tests.  A case is a dict of plain values:

  kind      "read"   one region of HiFi-like long reads, signed read graph, read voting
            "snp"    one region of ONT-like reads, SNP graph, refinement, parity swap
            "blocks" many phase blocks of uneven size in one graph (log-uniform 50-6,000
                     reads each), signed read graph
            "porec"  chromosome-like SNP graph: ONT-like reads and long-range Pore-C
                     contacts (CSR storage)
            "tiny"   80 index-placed reads (the smoke test's input)
            "product" one J x X product through the allocation-free BF16 entry point
  reads / snps / scale / blocks: the size;  R, T: replicas and bSB steps
  precision, variant, dt, check_every, patience, refine_max, linkage_k, schedule: options
  host      fragments in host memory, haplotypes back to host (else both on the device)
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2603_25762_gb300 import qhap, synth

PRECISION = {"fp32": qhap.PREC_FP32, "bf16": qhap.PREC_BF16, "bf16x2": qhap.PREC_BF16X2,
             "fp8": qhap.PREC_FP8}
BP_PER_READ = 4_000_000 / 7200   # HiFi-like regions: 27x of 15 kb reads
SNPS_PER_READ = 12_000 / 7200
BP_PER_ONT_READ = 4_000_000 / 3600  # ONT-like regions: 27x of 30 kb reads
SNPS_PER_ONT_READ = 12_000 / 3600


def listed():
    return [
        # the smallest call with the API's own defaults (FP32, 32 replicas): a single gene
        {"name": "tiny-fp32", "kind": "tiny", "R": 32, "T": 1000, "precision": "fp32"},
        # one J x X product of a half region through the allocation-free entry point
        {"name": "product-bf16", "kind": "product", "reads": 3001, "R": 512},
        # a gene cluster: a few row tiles, an odd read count, latency between steps
        {"name": "cluster-bf16", "kind": "read", "reads": 903, "R": 128, "T": 1000,
         "precision": "bf16"},
        # a 1 Mb window at a replica count that is an odd multiple of 64 (one launch a step)
        {"name": "window-bf16-r192", "kind": "read", "reads": 1801, "R": 192, "T": 500,
         "precision": "bf16"},
        # the benchmark's region: 7,200 reads x 1,024 replicas x 1,000 steps
        {"name": "region-bf16", "kind": "read", "reads": 7200, "R": 1024, "T": 1000,
         "precision": "bf16"},
        # the same region end to end from host buffers, with energy checks and early stop
        {"name": "region-bf16-stop-host", "kind": "read", "reads": 7200, "R": 1024, "T": 1000,
         "precision": "bf16", "check_every": 50, "patience": 3, "host": True},
        # the same region at the API's default precision
        {"name": "region-fp32", "kind": "read", "reads": 7200, "R": 256, "T": 500,
         "precision": "fp32"},
        # and with 8-bit operands
        {"name": "region-fp8", "kind": "read", "reads": 7200, "R": 512, "T": 500,
         "precision": "fp8"},
        # the SNP-based method on the benchmark's ONT-like region, refinement to its end
        {"name": "snp-region-bf16", "kind": "snp", "reads": 3600, "R": 512, "T": 2000,
         "precision": "bf16", "refine_max": 15},
        # a 1 Mb ONT window at the default precision, ragged replica count, lower linkage
        # depth
        {"name": "snp-window-fp32", "kind": "snp", "reads": 901, "R": 100, "T": 250,
         "precision": "fp32", "refine_max": 2, "linkage_k": 6},
        # many phase blocks of uneven size in one call
        {"name": "blocks-bf16", "kind": "blocks", "blocks": 96, "R": 256, "T": 1000,
         "precision": "bf16"},
        # a quarter chromosome with Pore-C contacts: long-range edges, CSR storage
        {"name": "porec-bf16", "kind": "porec", "scale": 0.25, "R": 128, "T": 400,
         "precision": "bf16", "refine_max": 2},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["read", "read", "read", "snp", "snp", "blocks", "porec", "product"])
    if kind == "product":
        reads = _log_int(rng, 60, 7200)
        return {"kind": kind, "reads": reads,
                "R": 64 * rng.randint(1, max(1, min(16, 4_194_304 // (reads + 256) // 64)))}
    if kind == "read":
        c = {"kind": kind, "reads": _log_int(rng, 60, 7200),
             "precision": rng.choice(["fp32", "bf16", "bf16", "fp8"])}
        if c["precision"] == "fp32":
            c["R"], c["T"] = _log_int(rng, 8, 256), _log_int(rng, 100, 500)
        else:
            c["R"] = 64 * _log_int(rng, 1, 16 if c["precision"] == "bf16" else 8)
            c["T"] = _log_int(rng, 100, 1000 if c["precision"] == "bf16" else 500)
        option = rng.choice(["", "", "stop", "discrete", "adiabatic", "host"])
        if option == "stop":
            c["check_every"], c["patience"] = rng.choice([25, 50, 100, 200]), rng.randint(2, 4)
        elif option == "discrete":
            c["variant"] = "discrete"
        elif option == "adiabatic":
            c["variant"], c["dt"] = "adiabatic", 0.1
        elif option == "host":
            c["host"] = True
        return c
    if kind == "snp":
        c = {"kind": kind, "precision": rng.choice(["fp32", "bf16", "bf16", "bf16x2"]),
             "refine_max": rng.randint(1, 3), "linkage_k": rng.choice([4, 6, 10])}
        if c["precision"] == "fp32":
            c["reads"], c["R"], c["T"] = _log_int(rng, 60, 900), _log_int(rng, 8, 128), \
                _log_int(rng, 50, 250)
        else:
            c["reads"], c["R"], c["T"] = _log_int(rng, 60, 3600), 64 * _log_int(rng, 1, 8), \
                _log_int(rng, 100, 1000)
        return c
    if kind == "blocks":
        c = {"kind": kind, "blocks": _log_int(rng, 4, 96),
             "precision": rng.choice(["fp32", "bf16", "bf16"])}
        if c["precision"] == "fp32":
            c["R"], c["T"] = _log_int(rng, 8, 64), _log_int(rng, 50, 200)
        else:
            c["R"], c["T"] = 64 * rng.randint(1, 4), _log_int(rng, 100, 1000)
        return c
    c = {"kind": "porec", "scale": round(math.exp(rng.uniform(math.log(0.04), math.log(0.25))), 4),
         "precision": rng.choice(["fp32", "bf16"]), "refine_max": rng.randint(1, 2)}
    if c["precision"] == "fp32":
        c["R"], c["T"] = 4 * rng.randint(2, 16), _log_int(rng, 25, 100)
    else:
        c["R"], c["T"] = 64 * rng.randint(1, 2), _log_int(rng, 50, 400)
    return c


def _blocks(n_blocks, seed):
    """Phase blocks laid end to end without shared SNPs: the benchmark's 50-6,000 reads at
    30x and 3 SNPs per kb.  The sizes are the log-uniform distribution's quantiles, in an
    order of the seed's (so that the totals do not depend on it)."""
    u = (np.random.default_rng(seed).permutation(n_blocks) + 0.5) / n_blocks
    ptr, cols, base, snps = [np.zeros(1, np.int64)], [], 0, 0
    for b, n in enumerate(np.rint(50 * 120.0 ** u).astype(int)):
        fr = synth.region_reads([seed, b], n_snps=round(1.5 * n), region=500 * int(n),
                                n_reads=int(n))
        ptr.append(fr.frag_ptr[1:] + base)
        cols.append((fr.snp + np.int32(snps), fr.allele, fr.qual, fr.is_porec))
        base += fr.nnz
        snps += fr.n_snps
    snp, allele, qual, porec = (np.concatenate(c) for c in zip(*cols))
    return synth.Fragments(snps, np.concatenate(ptr), snp, allele, qual, porec,
                           np.arange(snps), np.ones(snps, np.int8))


def _fragments(case, seed):
    kind = case["kind"]
    if kind == "tiny":
        return synth.tiny_reads(seed)
    if kind in ("read", "product"):
        n = case["reads"]
        return synth.region_reads(seed, n_snps=max(8, round(SNPS_PER_READ * n)),
                                  region=max(20_000, round(BP_PER_READ * n)), n_reads=n)
    if kind == "snp":
        n = case["reads"]
        return synth.region_reads(seed, n_snps=max(8, round(SNPS_PER_ONT_READ * n)),
                                  region=max(60_000, round(BP_PER_ONT_READ * n)), n_reads=n,
                                  len_mean=30_000, len_sd=20_000, len_max=150_000, flip_p=0.06,
                                  miss_p=0.0, qual=(7, 30), name="ont-region")
    if kind == "blocks":
        return _blocks(case["blocks"], seed)
    return synth.chromosome_porec(seed, scale=case["scale"])


_ctx = None


def _context():
    """One library context for the process, as a phasing program holds it."""
    global _ctx
    if _ctx is None:
        _ctx = qhap.Context(0)
    return _ctx


def prepare(case, seed):
    fr = _fragments(case, seed)
    cols = (fr.frag_ptr, fr.snp, fr.allele, fr.qual, fr.is_porec)
    snp = case["kind"] in ("snp", "porec")
    host = bool(case.get("host"))
    if host:  # pinned host buffers, as a read parser fills them
        held = [torch.from_numpy(np.ascontiguousarray(a)).pin_memory() for a in cols]
        arrays = (fr.n_snps,) + tuple(t.numpy() for t in held)
    else:
        held = None
        arrays = (fr.n_snps,) + tuple(torch.from_numpy(a).cuda() for a in cols)
    state = {"ctx": _context(), "arrays": arrays, "held": held, "host": host,
             "n_snps": fr.n_snps, "kind": case["kind"], "rows": case.get("blocks", 16),
             "graph": dict(mode=qhap.MODE_SNP if snp else qhap.MODE_READ,
                           linkage_k=case.get("linkage_k", 10))}
    if case["kind"] == "product":  # the graph is built once, the product runs many times
        torch.cuda.synchronize()
        g = state["ctx"].build_graph(arrays=arrays, on_device=True, **state["graph"])
        n_pad, pidx, _ = g.layout()
        gen = torch.Generator().manual_seed(seed)
        x = torch.zeros(case["R"], n_pad)
        live = torch.from_numpy(pidx[pidx >= 0].astype(np.int64))
        x[:, live] = 2 * torch.rand(case["R"], live.numel(), generator=gen) - 1
        state.update(g=g, R=case["R"], x=x.cuda(),
                     z=torch.zeros(case["R"], n_pad, device="cuda"))
        return state
    if not host:
        state["out"] = (torch.zeros(fr.n_snps, dtype=torch.int8, device="cuda"),
                        torch.zeros(fr.n_snps, dtype=torch.int8, device="cuda"),
                        torch.zeros(fr.n_snps, dtype=torch.int32, device="cuda"))
    state["solve"] = dict(replicas=case["R"], steps=case["T"], seed=1,
                          precision=PRECISION[case["precision"]],
                          refine_max=case.get("refine_max", 15),
                          variant=case.get("variant", "ballistic"), dt=case.get("dt", 1.0),
                          check_every=case.get("check_every", 0),
                          patience=case.get("patience", 0))
    return state


def run(state):
    ctx = state["ctx"]
    if state["kind"] == "product":
        ctx.matvec_bf16_noalloc(state["g"], state["R"], state["x"], state["z"])
        return state["z"]
    g = ctx.build_graph(arrays=state["arrays"], on_device=not state["host"], **state["graph"])
    sol = ctx.solve(g, **state["solve"])
    hap1, hap2, block_id = ctx.phase(g, sol, state["n_snps"],
                                     out=None if state["host"] else state["out"])
    # every replica's cut of each block, in as many rows for every seed (a region of reads
    # is one to a few blocks)
    cuts = np.zeros((state["rows"], state["solve"]["replicas"]))
    rows = min(g.n_blocks, state["rows"])
    cuts[:rows] = sol.cuts()[:rows]
    got = {"hap1": hap1, "hap2": hap2, "block_id": block_id, "spins": sol.spins(g.n_nodes),
           "cuts": cuts}
    sol.free()
    g.free()
    return got


# mean stored edges per vertex of the generators' graphs (both directions counted)
def _degree(case):
    if case["kind"] == "tiny":
        return 10.5
    if case["kind"] in ("read", "product"):
        return min(53.0, case["reads"] - 1.0)
    if case["kind"] == "snp":
        return min(468.0, SNPS_PER_ONT_READ * case["reads"] - 1.0)
    return 59.0 if case["kind"] == "blocks" else 215.0


def work(case):
    """Fragments read once, results written once; the product and the update of every spin
    of one solve (a refinement that goes on repeats them: counted once)."""
    kind = case["kind"]
    if kind == "tiny":
        frags, snps, entries, nodes, blocks = 80, 300, 1600, 80, 1
    elif kind in ("read", "product"):
        frags = case["reads"]
        snps, entries, nodes, blocks = SNPS_PER_READ * frags, 44 * frags, frags, 1
    elif kind == "snp":
        frags = case["reads"]
        snps, entries, blocks = SNPS_PER_ONT_READ * frags, 88 * frags, 1
        nodes = snps
    elif kind == "blocks":
        blocks = case["blocks"]
        frags = 1243 * blocks  # mean of exp(U(ln 50, ln 6000))
        snps, entries, nodes = 1.5 * frags, 44 * frags, frags
    else:
        frags, snps = 2_250_000 * case["scale"], 200_000 * case["scale"]
        entries, nodes, blocks = 13_000_000 * case["scale"], snps, 1
    edges = nodes * _degree(case)
    R = case["R"]
    if kind == "product":  # J (2 B), x and z (4 B each)
        return {"bytes": 2 * edges + 8 * nodes * R, "flops": 2 * edges * R}
    io = 8 * frags + 6 * entries + frags + 6 * snps + nodes + 8 * blocks * R
    return {"bytes": io, "flops": (2 * edges + 8 * nodes) * R * case["T"]}


def exact(case, seed):
    """The product J x X in 64 bits: J = M M^T off the diagonal (signed read graph), X as
    the BF16 operand holds it, at the padded position of each read (blocks numbered by
    their smallest read, single reads dropped, each block padded to 128).  A whole solve's
    trajectories are chaotic: it has no 64-bit value to hold them to."""
    if case["kind"] != "product":
        return None
    fr = _fragments(case, seed)
    m = fr.n_frags
    rid = np.repeat(np.arange(m), np.diff(fr.frag_ptr))
    M = torch.zeros(m, fr.n_snps, dtype=torch.float64)
    M[rid, fr.snp.astype(np.int64)] = torch.from_numpy(fr.allele.astype(np.float64))
    M = M.cuda()
    J = M @ M.T
    J.fill_diagonal_(0)
    label = torch.arange(m, device="cuda")
    edge = J != 0
    while True:  # smallest label of the neighbourhood until nothing changes
        near = torch.where(edge, label[None, :], m).amin(dim=1)
        new = torch.minimum(label, near)
        new = new[new]
        if bool((new == label).all()):
            break
        label = new
    label = label.cpu().numpy()
    pos, at = np.full(m, -1, np.int64), 0
    for root in np.unique(label):
        members = np.flatnonzero(label == root)
        if members.size < 2:
            continue
        pos[members] = at + np.arange(members.size)
        at += (members.size + 127) // 128 * 128
    live = np.flatnonzero(pos >= 0)
    gen = torch.Generator().manual_seed(seed)
    X = torch.zeros(case["R"], m, dtype=torch.float64)
    # prepare() draws x in the order of the live reads
    X[:, live] = (2 * torch.rand(case["R"], live.size, generator=gen) - 1).bfloat16().double()
    Z = torch.zeros(case["R"], at, dtype=torch.float64, device="cuda")
    Z[:, torch.from_numpy(pos[live]).cuda()] = (X.cuda() @ J)[:, torch.from_numpy(live).cuda()]
    return Z
