"""Timed cases: what a program that searches a protein database has this
library do, through its public entry points.

A case names one kind of call, the model lengths it scores and the database it
scores them against.  Databases are background residues with lognormal
lengths, some with planted homologous segments or a tail of very long
sequences; profiles are realistic ones (``synth.make_profile``,
``synth.make_vit_profile``).

Kinds:
  request   a batch of queries scored with both filters into host buffers
            (``scan_batch``): one search request answered at once
  scan      plain one-query scans, MSV then SSV, into device buffers
            (``msv_scan``, ``ssv_scan``)
  plans     a batch of queries as one graph-captured plan per filter
  one_sweep a batch of queries as one plan that gives both filters
  stages    the pipeline: SSV over the database, MSV and then the gapped
            Viterbi filter over the survivors (``pipeline_scan``,
            ``viterbi_rescore``)
  viterbi   the gapped Viterbi filter over every sequence (``viterbi_scan``)
"""
import math

import numpy as np
import torch

from paper_1707_09683_gb300 import mpf, synth


def listed():
    base = dict(mean=355, max_len=35000, tail=0.0, planted=0.0)

    def case(name, kind, Ms, n_seqs, **kw):
        return dict(base, name=name, kind=kind, Ms=" ".join(map(str, Ms)), n_seqs=n_seqs, **kw)

    sweep = [48, 100, 200, 400, 800, 1600, 2405]
    return [
        # A single query answered against a small in-house collection: launch
        # and copy latency.
        case("request_m100_1k", "request", [100], 1000),
        # The plain one-query workload: one short domain, a bacterial-size
        # proteome.
        case("scan_m100_10k", "scan", [100], 10000, mean=350, max_len=5000),
        # An average protein-length model against a larger database.
        case("scan_m400_100k", "scan", [400], 100000),
        # The longest model of the length sweep.
        case("scan_m2405_60k", "scan", [2405], 60000),
        # A whole-genome set: few sequences, some of them titin-sized.
        case("scan_m777_tail", "scan", [777], 6001, tail=0.002),
        # The length sweep as captured plans, as a batch service runs it.
        case("plans_sweep_100k", "plans", sweep, 100000),
        # A mixed batch with homologues (overflows, exact rescoring), both
        # filters from one sweep of the database.
        case("one_sweep_16q_50k", "one_sweep",
             [1937, 811, 63, 1290, 399, 2211, 1022, 150, 702, 1675, 288, 2499, 517, 931, 1403, 87],
             50000, mean=270, planted=0.05),
        # A model past the striped table (giant multi-domain protein).
        case("one_sweep_m5000_20k", "one_sweep", [5000], 20000),
        # The three-stage pipeline, about 2% of the sequences passing.
        case("stages_sweep_80k", "stages", sweep, 80000),
        # The Viterbi filter by itself: a short model on few sequences, an
        # average one and the longest one of the sweep on many.
        case("viterbi_m150_1k", "viterbi", [150], 1003),
        case("viterbi_m400_20k", "viterbi", [400], 20000),
        case("viterbi_m2405_20k", "viterbi", [2405], 20000),
    ]


def draw(rng):
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["request", "scan", "scan", "plans", "one_sweep", "stages", "viterbi", "viterbi"])
    planted = tail = 0.0
    if kind == "request":
        Ms, n = [log_int(48, 2405) for _ in range(rng.randint(1, 4))], log_int(300, 10000)
    elif kind == "scan":
        Ms, n = [log_int(30, 2500)], log_int(1000, 100000)
        tail = rng.choice([0.0, 0.0, 0.001])
        planted = rng.choice([0.0, 0.02])
    elif kind == "plans":
        Ms, n = [log_int(48, 2405) for _ in range(rng.randint(2, 9))], log_int(5000, 60000)
    elif kind == "one_sweep":
        if rng.random() < 0.4:
            Ms, n = [rng.randint(3073, 9000)], log_int(2000, 20000)
        else:
            Ms, n = [rng.randint(50, 2500) for _ in range(rng.randint(2, 12))], log_int(5000, 50000)
            planted = 0.05
    elif kind == "stages":
        Ms, n = [log_int(48, 2405) for _ in range(rng.randint(1, 7))], log_int(10000, 80000)
        planted = rng.choice([0.0, 0.02])
    else:
        Ms, n = [log_int(40, 2700)], log_int(500, 20000)
    return dict(kind=kind, Ms=" ".join(map(str, Ms)), n_seqs=n, mean=rng.randint(200, 400),
                max_len=35000, tail=tail, planted=planted)


FILTER_PASS = 0.02      # fraction of the sequences that pass a pipeline stage


def _lengths(case):
    return [int(m) for m in case["Ms"].split()]


def _inputs(case, seed):
    """Host inputs: profile records, Viterbi profile records, database."""
    r_prof, r_db, r_plant = [np.random.Generator(np.random.PCG64(s))
                             for s in np.random.SeedSequence(int(seed)).spawn(3)]
    Ms = _lengths(case)
    profs = [synth.make_profile(M, r_prof) for M in Ms] if case["kind"] != "viterbi" else []
    vits = [synth.make_vit_profile(M, r_prof) for M in Ms] if case["kind"] in ("viterbi", "stages") else []
    db = synth.make_database(case["n_seqs"], case["mean"], 10, case["max_len"], r_db, tail_frac=case["tail"])
    if case["planted"]:
        synth.plant_segments(db, profs, case["planted"], r_plant)
    return profs, vits, db


def prepare(case, seed):
    kind, n, nq = case["kind"], case["n_seqs"], len(_lengths(case))
    profs, vits, db = _inputs(case, seed)
    ctx = mpf.Context(0)
    st = {"kind": kind, "ctx": ctx, "stream": ctx.torch_stream(),
          "db": mpf.Database(ctx, db.residues, db.offsets, db.lengths),
          "profs": [mpf.Profile(ctx, p) for p in profs], "vits": [mpf.VitProfile(ctx, v) for v in vits]}

    def buffers(count, types=(torch.uint8, torch.uint8, torch.float32)):
        return [torch.zeros(count, dtype=t, device="cuda") for t in types]

    if kind == "request":
        st["out"] = [np.zeros(2 * nq * n, dtype=t) for t in (np.uint8, np.uint8, np.float32)]
    elif kind == "scan":
        st["out"] = buffers(n) + buffers(n)
    elif kind == "plans":
        st["out"] = buffers(nq * n) + buffers(nq * n)
        torch.cuda.synchronize()
        st["plans"] = [mpf.Plan(ctx, f, st["profs"], st["db"], *st["out"][3 * f:3 * f + 3])
                       for f in (mpf.MSV, mpf.SSV)]
        for plan in st["plans"]:
            plan.capture_graph()
    elif kind == "one_sweep":
        st["out"] = buffers(2 * nq * n)
        torch.cuda.synchronize()
        st["plans"] = [mpf.Plan(ctx, mpf.MSV_SSV, st["profs"], st["db"], *st["out"])]
        st["plans"][0].capture_graph()
    elif kind == "stages":
        vit_types = (torch.int16, torch.uint8, torch.float32)
        count = lambda: torch.zeros(nq, dtype=torch.int32, device="cuda")  # noqa: E731
        st["out"] = buffers(nq * n) + buffers(nq * n) + [count()] + buffers(nq * n, vit_types) + [count()]
        # The pass score, calibrated once on the program's own database.
        torch.cuda.synchronize()
        mpf.scan_batch(ctx, mpf.SSV, st["profs"], st["db"], *st["out"][:3])
        ctx.sync()
        st["min_nat"] = float(torch.quantile(st["out"][2][:1 << 20].double(), 1.0 - FILTER_PASS))
    else:
        st["out"] = buffers(nq * n, (torch.int16, torch.uint8, torch.float32))
    torch.cuda.synchronize()
    return st


def run(state):
    ctx, db, out, kind = state["ctx"], state["db"], state["out"], state["kind"]
    if kind == "request":
        mpf.scan_batch(ctx, mpf.MSV_SSV, state["profs"], db, *out)
        return out
    if kind == "scan":
        mpf.msv_scan(ctx, state["profs"][0], db, *out[:3])
        mpf.ssv_scan(ctx, state["profs"][0], db, *out[3:])
    elif kind in ("plans", "one_sweep"):
        for plan in state["plans"]:
            plan.launch()
    elif kind == "stages":
        mpf.pipeline_scan(ctx, state["profs"], db, state["min_nat"], out[0:3], out[3:6], out[6])
        mpf.viterbi_rescore(ctx, state["vits"], db, out[4], out[5], state["min_nat"], *out[7:10], out[10])
    else:
        mpf.viterbi_scan(ctx, state["vits"], db, *out)
    # The results are ready for the caller's stream (no host wait).
    torch.cuda.current_stream().wait_stream(state["stream"])
    return out


def work(case):
    kind, n, Ms = case["kind"], case["n_seqs"], _lengths(case)
    residues = n * case["mean"]
    if case["tail"]:
        residues += int(n * case["tail"] * 30000 / math.log(7.0))   # mean of a log-uniform 5,000-35,000
    nq, cells = len(Ms), sum(Ms) * residues
    # Byte filters: add, restart at zero and running maximum per cell, one
    # sweep for both filters.  Viterbi: 8 adds and 7 maxima per cell.
    if kind == "viterbi":
        return {"bytes": residues + 12 * n + nq * n * 7 + sum(Ms) * (20 + 8) * 2, "flops": 15 * cells}
    if kind == "stages":
        return {"bytes": residues + 12 * n + nq * n * 19 + sum(Ms) * (20 + 28 * 2),
                "flops": int(cells * (3 + FILTER_PASS * (3 + 15)))}
    return {"bytes": residues + 12 * n + 2 * nq * n * 6 + sum(Ms) * 20, "flops": 3 * cells}


# ---------------------------------------------------------------------------
# The recurrences in 64-bit integers (torch), written out plainly: nodes along
# the last axis, sequences sorted longest first so that the rows still
# running are a prefix.

EXACT_MAX_CELLS = 2.2e11


def _rows(db, M):
    """Chunks of sequences (longest first): their numbers, their lengths and
    their residues by row, zero past a sequence's end."""
    order = np.argsort(-db.lengths.astype(np.int64), kind="stable")
    dev = torch.device("cuda")
    res = torch.from_numpy(db.residues).to(dev)
    off, length = db.offsets.astype(np.int64), db.lengths.astype(np.int64)
    per = max(1, (1 << 25) // M)
    for s in range(0, order.size, per):
        idx = order[s:s + per]
        o, L = torch.from_numpy(off[idx]).to(dev), torch.from_numpy(length[idx]).to(dev)
        left = np.searchsorted(-length[idx], -np.arange(int(length[idx][0])), side="left")   # lengths above row i

        def codes(i, a, o=o):
            return res[o[:a] + i].long()
        yield torch.from_numpy(idx).to(dev), L, left, codes


def _exact_bytes(prof, db):
    """(raw, flag, nat) of MSV and of SSV for every sequence."""
    dev = torch.device("cuda")
    n, M = db.n_seqs, prof.M
    cost = torch.from_numpy(prof.cost).to(dev).long()
    tjb = torch.from_numpy(prof.tjb_by_len).to(dev).long()
    outs = [[torch.zeros(n, dtype=t, device=dev) for t in (torch.uint8, torch.uint8, torch.float64)] for _ in range(2)]
    for idx, L, left, codes in _rows(db, M):
        m = idx.numel()
        t = tjb[L.clamp(max=tjb.numel() - 1)]
        xB = (prof.base - (t + prof.tbm)).clamp(0, 255)
        xJ, over = torch.zeros_like(xB), torch.zeros(m, dtype=torch.bool, device=dev)
        R = torch.zeros_like(xB)
        dp = torch.zeros(m, M, dtype=torch.int64, device=dev)
        r = torch.zeros_like(dp)
        for i, a in enumerate(left):
            a = int(a)
            c = cost[codes(i, a)]
            prev = torch.nn.functional.pad(dp[:a, :-1], (1, 0))
            d = (torch.maximum(prev, xB[:a, None]) + prof.bias).clamp_(0, 255).sub_(c).clamp_(0, 255)
            dp[:a] = d
            xE = d.amax(1)
            over[:a] |= xE >= 255 - prof.bias
            xJ[:a] = torch.maximum(xJ[:a], (xE - prof.tec).clamp(0, 255))
            xB[:a] = (xJ[:a].clamp(min=prof.base) - (t[:a] + prof.tbm)).clamp(0, 255)
            s = (torch.nn.functional.pad(r[:a, :-1], (1, 0)) + prof.bias).sub_(c).clamp_(0, 255)
            r[:a] = s
            R[:a] = torch.maximum(R[:a], s.amax(1))
        inf = torch.full((), math.inf, dtype=torch.float64, device=dev)
        for (raw, flag, nat), score, ovf, num in (
                (outs[0], xJ, over, xJ - t - prof.base),
                (outs[1], R, R == 255, R - prof.tbm - prof.tec - 2 * t)):
            raw[idx] = torch.where(ovf, 255, score).to(torch.uint8)
            flag[idx] = ovf.to(torch.uint8)
            nat[idx] = torch.where(ovf, inf, num.double() / prof.scale - 3.0)
    return outs


def _exact_viterbi(vp, db, keep=None):
    """(score, flag, nat) of the Viterbi filter for every sequence (or the
    sequences of the mask ``keep``; the others read as filtered).  Delete
    scores: with moves <= 0 the saturating chain is the larger of -32768 and
    the unsaturated one, a running maximum of M - (sum of D->D moves)."""
    dev = torch.device("cuda")
    LOW = -32768
    if keep is None:
        score, flag, nat = [torch.zeros(db.n_seqs, dtype=t, device=dev) for t in (torch.int16, torch.uint8, torch.float64)]
        sub, back = db, None
    else:
        score = torch.full((db.n_seqs,), LOW, dtype=torch.int16, device=dev)
        flag = torch.full((db.n_seqs,), 2, dtype=torch.uint8, device=dev)
        nat = torch.full((db.n_seqs,), math.nan, dtype=torch.float64, device=dev)
        back = torch.nonzero(keep).flatten()
        if back.numel() == 0:
            return [score, flag, nat]
        pick = back.cpu().numpy()
        sub = synth.Database(residues=db.residues, offsets=db.offsets[pick], lengths=db.lengths[pick])
    msc = torch.from_numpy(vp.msc).to(dev).long()
    BM, MM, IM, DM, MI, II, MD, DD = torch.from_numpy(vp.trans).to(dev).long()
    NN, NB, EC, CC, CT, EJ, JJ, JB = [int(v) for v in vp.special]
    DDs = DD.clone()
    DDs[:2] = 0                              # D_1 does not exist
    P = torch.cumsum(DDs, 0)                 # sum of the D->D moves up to each node

    def sat(v):
        return v.clamp(LOW, 32767)

    def before(v):                           # node k - 1; nothing before node 1
        return torch.nn.functional.pad(v[:, :-1], (1, 0), value=LOW)

    for idx, L, left, codes in _rows(sub, vp.M):
        m = idx.numel()
        Mr = torch.full((m, vp.M), LOW, dtype=torch.int64, device=dev)
        Ir, Dr = Mr.clone(), Mr.clone()
        xN = torch.full((m,), vp.base, dtype=torch.int64, device=dev)
        xB = sat(xN + NB)
        xJ, xC = torch.full_like(xN, LOW), torch.full_like(xN, LOW)
        over = torch.zeros(m, dtype=torch.bool, device=dev)
        for i, a in enumerate(left):
            a = int(a)
            best = torch.maximum(torch.maximum(before(Mr[:a]) + MM, before(Ir[:a]) + IM),
                                 torch.maximum(before(Dr[:a]) + DM, xB[:a, None] + BM))
            I = sat(torch.maximum(Mr[:a] + MI, Ir[:a] + II))
            I[:, -1] = LOW
            Mn = sat(sat(best) + msc[codes(i, a)])
            D = sat(before(Mn) + MD)
            D[:, 0] = LOW
            D = (torch.cummax(D - P, 1).values + P).clamp_(min=LOW)
            Mr[:a], Ir[:a], Dr[:a] = Mn, I, D
            xE = torch.maximum(Mn, D).amax(1)
            over[:a] |= xE >= 32767
            xN[:a] = sat(xN[:a] + NN)
            xC[:a] = torch.maximum(sat(xC[:a] + CC), sat(xE + EC))
            xJ[:a] = torch.maximum(sat(xJ[:a] + JJ), sat(xE + EJ))
            xB[:a] = torch.maximum(sat(xN[:a] + NB), sat(xJ[:a] + JB))
        to = idx if back is None else back[idx]
        sc = torch.where(over, 32767, sat(xC + CT))
        score[to], flag[to] = sc.to(torch.int16), over.to(torch.uint8)
        inf = torch.full((), math.inf, dtype=torch.float64, device=dev)
        nat[to] = torch.where(over, inf, (sc - vp.base).double() / vp.scale - 3.0)
    return [score, flag, nat]


def exact(case, seed):
    kind, n = case["kind"], case["n_seqs"]
    if work(case)["flops"] > EXACT_MAX_CELLS * (15 if kind == "viterbi" else 3):
        return None
    profs, vits, db = _inputs(case, seed)
    if kind == "viterbi":
        return _exact_viterbi(vits[0], db)
    both = [_exact_bytes(p, db) for p in profs]
    msv, ssv = [[torch.cat([q[f][j] for q in both]) for j in range(3)] for f in range(2)]
    if kind in ("request", "one_sweep"):
        out = [torch.cat([msv[j], ssv[j]]) for j in range(3)]
        return [v.cpu().numpy() for v in out] if kind == "request" else out
    if kind in ("scan", "plans"):
        return msv + ssv
    # The pass score is compared with single-precision scores.
    min_nat = float(torch.quantile(ssv[2].float()[:1 << 20].double(), 1.0 - FILTER_PASS))
    passed = (ssv[1] == 1) | (ssv[2].float() >= min_nat)
    m = [torch.where(passed, msv[0], 0), torch.where(passed, msv[1], 2),
         torch.where(passed, msv[2], math.nan)]
    keep = (m[1] == 1) | ((m[1] == 0) & (m[2].float() >= min_nat))
    v = [_exact_viterbi(vp, db, keep[q * n:(q + 1) * n]) for q, vp in enumerate(vits)]
    counts = [x.view(-1, n).sum(1).to(torch.int32) for x in (passed, keep)]
    return ssv + m + [counts[0]] + [torch.cat([q[j] for q in v]) for j in range(3)] + [counts[1]]
