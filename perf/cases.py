"""Timed cases of the framework: calls that its users make, through its public entry points.

Inputs are synthetic proteomes of the recipe the benchmark uses (planted families of members
with 30 % substitutions and 5 % indels, lognormal root lengths of median 350 clipped to
30-5,000, singletons), made from the seed alone; tandem repeats stand in for the long tail.
Every case names its `kind`; `draw` gives cases of the same kinds with other sizes and options.
"""
import math

import numpy as np
import torch

import paper_1908_10574_gb300 as cm
from paper_1908_10574_gb300 import synth

GAP_OPEN, GAP_EXTEND = 11, 1
T, M_T, M_U = 100, 138, 15             # BLOSUM62 thresholds of the clustering runs
T_PAM, M_T_PAM = 181, 250              # the paper's, for PAM250
_DEVICE = "cuda" if torch.cuda.is_available() else "cpu"


def listed():
    return [
        # one query looked up in a small family collection: the smallest call, all latency
        {"name": "search_200", "kind": "search", "queries": 1, "subjects": 200,
         "alphabet": 20, "device": False},
        # labelling of ranker training pairs: pairs inside groups of 128 proteins, few per query
        {"name": "pairs_50k", "kind": "pairs", "proteins": 5000, "group": 128, "pairs": 50000,
         "alphabet": 20, "device": True},
        # scores of long tandem repeats beyond the int16 range (the long tail of a proteome)
        {"name": "long_repeats", "kind": "long", "pairs": 24, "lo": 8000, "hi": 12000},
        # all-against-all of the small family set, as text under PAM250 with 24 letters
        {"name": "allpairs_200_ascii", "kind": "allpairs", "proteins": 200, "parts": 1,
         "alphabet": 24, "ascii": True, "device": False},
        # the headline: one sixteenth of the all-against-all of 20,000 proteins
        {"name": "allpairs_20k_part", "kind": "allpairs", "proteins": 20000, "parts": 16,
         "alphabet": 20, "ascii": False, "device": True},
        # alignment cells of similar pairs (the transitivity test's input)
        {"name": "cells_20k", "kind": "cells", "proteins": 20000, "pairs": 20000,
         "alphabet": 20, "device": False},
        # the same without allocation, as a resident service calls it
        {"name": "cells_noalloc_200", "kind": "noalloc", "proteins": 400, "pairs": 200, "longest": 600},
        # tracebacks of the similar pairs a clustering reports
        {"name": "align_2k", "kind": "align", "proteins": 4000, "pairs": 2000, "alphabet": 20,
         "longest": 1500},
        # ranker embeddings of a set (inference before a ranked merge)
        {"name": "embed_4k", "kind": "embed", "proteins": 4000, "pairs": 0},
        # loss and gradient of one training batch
        {"name": "loss_grad_128", "kind": "grad", "proteins": 128, "pairs": 1280},
        # ranker training from given weights: one epoch, one group of 128 proteins per step
        {"name": "train_1280", "kind": "train", "proteins": 1280, "group": 128, "pairs": 12800},
        # whole clustering
        {"name": "cluster_merge_3k", "kind": "cluster", "proteins": 3000, "mode": "plain",
         "alphabet": 20},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["search", "pairs", "long", "allpairs", "allpairs", "cells", "noalloc",
                       "align", "embed", "grad", "train", "cluster"])
    c = {"kind": kind}
    alphabet = rng.choice([20, 20, 24])
    if kind == "search":
        c.update(queries=_log(rng, 1, 16), subjects=_log(rng, 20, 2000), alphabet=alphabet,
                 device=rng.random() < 0.5)
    elif kind == "pairs":
        n = _log(rng, 100, 5000)
        c.update(proteins=n, group=rng.randint(32, 200), pairs=n * rng.randint(2, 10),
                 alphabet=alphabet, device=rng.random() < 0.5)
    elif kind == "long":
        lo = _log(rng, 2500, 8000)
        c.update(pairs=rng.randint(2, 24), lo=lo, hi=lo + rng.randint(10, 4000))
    elif kind == "allpairs":
        n = _log(rng, 30, 20000)
        parts = max(1, math.ceil(16 * (n / 20000.0) ** 2)) * rng.choice([1, 1, 2])
        c.update(proteins=n, parts=parts, alphabet=alphabet, ascii=rng.random() < 0.3,
                 device=rng.random() < 0.5)
    elif kind == "cells":
        n = _log(rng, 50, 20000)
        c.update(proteins=n, pairs=n, alphabet=alphabet, device=rng.random() < 0.3)
    elif kind == "noalloc":
        n = _log(rng, 16, 500)
        c.update(proteins=2 * n, pairs=n, longest=_log(rng, 100, 1000))
    elif kind == "align":
        n = _log(rng, 20, 2000)
        c.update(proteins=2 * n + 20, pairs=n, alphabet=alphabet, longest=_log(rng, 300, 3000))
    elif kind == "embed":
        n = _log(rng, 20, 4000)
        c.update(proteins=n, pairs=rng.choice([0, 5 * n]))
    elif kind == "grad":
        n = _log(rng, 16, 500)
        c.update(proteins=n, pairs=n * rng.randint(3, 12))
    elif kind == "train":
        g = rng.randint(48, 160)
        c.update(proteins=g * rng.randint(3, 10), group=g)
        c.update(pairs=10 * c["proteins"])
    else:
        c.update(proteins=_log(rng, 100, 3000), alphabet=alphabet,
                 mode=rng.choice(["plain", "plain", "partial", "greedy"]))
    return c


# ---- inputs ---------------------------------------------------------------------------------
_QUANTILE = np.searchsorted(np.cumsum(synth.BACKGROUND), (np.arange(65536) + 0.5) / 65536.0,
                            side="right").clip(0, 19).astype(np.uint8)


def _residues(rng, n):
    return _QUANTILE[rng.integers(0, 65536, size=n, dtype=np.uint16)]


def _proteome(rng, n, family=8, singles=0.2, alphabet=20, longest=5000):
    """SeqSet of n proteins: families of `family` plus a fraction of singletons, shuffled."""
    n_single = min(n, int(round(n * singles)))
    n_fam = -(-(n - n_single) // family)
    fam = np.concatenate([np.repeat(np.arange(n_fam), family)[:n - n_single],
                          n_fam + np.arange(n_single)])
    roots = synth.lognormal_lengths(rng, n_fam + n_single, hi=longest)
    roff = np.concatenate([[0], np.cumsum(roots)])
    root = _residues(rng, int(roff[-1]))
    fam = fam[rng.permutation(n)]
    lens = roots[fam]
    off = np.concatenate([[0], np.cumsum(lens)])
    seq = root[np.arange(off[-1]) - np.repeat(off[:-1] - roff[fam], lens)]
    # per residue: substitution, or a single-residue deletion or insertion
    u = rng.random(len(seq), dtype=np.float32)
    sub = u < 0.30
    new = _residues(rng, int(sub.sum()))
    old = seq[sub]
    seq[sub] = np.where(new == old, (old + 1) % 20, new)
    ev = rng.random(len(seq), dtype=np.float32)
    counts = np.ones(len(seq), np.int8)
    counts[ev < 0.025] = 0
    counts[ev > 0.975] = 2
    counts[off[:-1]] = 1                                  # no protein vanishes
    out = np.repeat(seq, counts)
    pos = np.cumsum(counts, dtype=np.int64)
    ins = pos[counts == 2] - 2
    out[ins] = _residues(rng, len(ins))
    noff = np.concatenate([[0], pos[off[1:] - 1]]).astype(np.int64)
    if alphabet == 24:                                    # ambiguity letters, one in 200
        amb = rng.integers(0, len(out), size=len(out) // 200)
        out[amb] = rng.choice(np.array([20, 21, 22], np.uint8), size=len(amb))
    return synth.SeqSet(out, noff, fam)


def _family_pairs(rng, family, n):
    """n pairs of two members of one family, and a tenth of unrelated ones."""
    order = np.argsort(family, kind="stable")
    f = family[order]
    start = np.searchsorted(f, f, side="left")
    size = np.searchsorted(f, f, side="right") - start
    multi = np.flatnonzero(size > 1)
    a = rng.choice(multi, size=n) if len(multi) else rng.integers(0, len(f), size=n)
    b = start[a] + (a - start[a] + 1 + rng.integers(0, np.maximum(size[a] - 1, 1))) % size[a]
    far = rng.random(n) < 0.1
    b = np.where(far, rng.integers(0, len(f), size=n), b)
    return np.stack([order[a], order[b]], 1).astype(np.int32)


def _group_pairs(rng, family, n, group):
    """n pairs inside groups of `group` proteins dealt family by family: half of them within
    a family, half drawn uniformly in the group; with the group's label as 0/1 relation."""
    order = np.argsort(family, kind="stable")
    f = family[order]
    a = rng.integers(0, len(f), size=n)
    g0 = a // group * group
    b = g0 + rng.integers(0, np.minimum(group, len(f) - g0))
    start = np.searchsorted(f, f, side="left")
    size = np.searchsorted(f, f, side="right") - start
    near = start[a] + rng.integers(0, size[a])
    b = np.where((rng.random(n) < 0.5) & (size[a] > 1) & (near // group == a // group), near, b)
    b = np.where(b == a, g0 + (b - g0 + 1) % np.minimum(group, len(f) - g0), b)
    pairs = np.stack([order[a], order[b]], 1).astype(np.int32)
    return pairs, (f[a] == f[b]).astype(np.float32)


_LETTERS = np.frombuffer(synth.ALPHABET24.encode(), np.uint8)


def _matrix(case):
    return synth.PAM250_24 if case.get("alphabet") == 24 else synth.BLOSUM62


def _params(rng):
    """Ranker weights at their initialisation's scale, small biases."""
    parts = [rng.standard_normal(20 * 32), rng.standard_normal(9 * 32 * 128) * (2 / 288) ** 0.5,
             rng.standard_normal(128) * 0.05, rng.standard_normal(9 * 128 * 128) * (2 / 1152) ** 0.5,
             rng.standard_normal(128) * 0.05, rng.standard_normal(9 * 128 * 128) * (1 / 1152) ** 0.5,
             rng.standard_normal(128) * 0.05, np.array([10.0, -2.0])]
    return np.concatenate(parts).astype(np.float32)


def _inputs(case, seed):
    """Host arrays of a case, from the seed alone."""
    rng = np.random.default_rng([1908, int(seed)])
    kind, s = case["kind"], {}
    if kind == "search":
        ss = _proteome(rng, case["subjects"] + case["queries"], alphabet=case["alphabet"])
        q = np.arange(case["queries"], dtype=np.int32)
        t = np.arange(case["subjects"], dtype=np.int32) + case["queries"]
        s["pairs"] = np.stack([np.repeat(q, len(t)), np.tile(t, len(q))], 1).astype(np.int32)
    elif kind == "pairs":
        ss = _proteome(rng, case["proteins"], alphabet=case["alphabet"])
        s["pairs"], _ = _group_pairs(rng, ss.family, case["pairs"], case["group"])
    elif kind == "long":
        n = max(2, case["pairs"] // 2)
        motifs = [_residues(rng, 40) for _ in range(2)]
        ss = synth.SeqSet.from_list([
            synth.tandem_repeat(rng, int(rng.integers(case["lo"], case["hi"] + 1)),
                                motif=motifs[i % 2]) for i in range(n)])
        i, j = np.triu_indices(n, 1)
        take = rng.permutation(len(i))[:case["pairs"]]
        s["pairs"] = np.stack([i[take], j[take]], 1).astype(np.int32)
    elif kind in ("allpairs", "cluster"):
        fam, single = (10, 0.0) if kind == "allpairs" else (8, 0.2)
        ss = _proteome(rng, case["proteins"], fam, single, case["alphabet"])
    elif kind in ("cells", "align", "noalloc"):
        ss = _proteome(rng, case["proteins"], alphabet=case.get("alphabet", 20),
                       longest=case.get("longest", 5000))
        s["pairs"] = _family_pairs(rng, ss.family, case["pairs"])
    elif kind == "embed":
        ss = _proteome(rng, case["proteins"])
        s["params"] = _params(rng)
        if case["pairs"]:
            s["pairs"] = rng.integers(0, len(ss), size=(case["pairs"], 2)).astype(np.int32)
    else:
        ss = _proteome(rng, case["proteins"])
        s["params"] = _params(rng)
        s["pairs"], s["labels"] = _group_pairs(rng, ss.family, case["pairs"],
                                               case.get("group", case["proteins"]))
    s["seqs"], s["offsets"] = ss.seqs, ss.offsets
    if kind == "train":
        _standardize(s)
    return s


def _standardize(s):
    """Rescales W3 and b3 so that every channel of the pooled vectors has zero mean and unit
    variance over some sequences, as a program does before it trains."""
    v, _, _ = _forward64(s, torch.from_numpy(s["params"].astype(np.float64)).to(_DEVICE),
                         np.arange(min(64, len(s["offsets"]) - 1)))
    v = v.cpu().numpy()
    mean, sd = v.mean(0), v.std(0, ddof=1) + 1e-6
    w3, b3 = s["params"][-2 - 128 - 9 * 128 * 128:-2 - 128], s["params"][-2 - 128:-2]
    w3[:] = (w3.reshape(-1, 128) / sd).ravel()
    b3[:] = (b3 - mean) / sd


_ALIGN_RUNS = 200                      # room for the runs of one traceback, on average


def _padded(a, rows, fill=-1):
    """Results of as many rows as the data give, in an array of a fixed number of rows."""
    out = np.full((rows,) + a.shape[1:], fill, a.dtype)
    out[:len(a)] = a
    return out


def prepare(case, seed):
    s = _inputs(case, seed)
    s["case"] = case
    s["matrix"] = _matrix(case)
    if case.get("ascii"):
        s["seqs"] = _LETTERS[s["seqs"]]
    if case.get("device") or case["kind"] == "noalloc":
        for k in ("seqs", "offsets", "pairs"):
            if k in s:
                s[k] = torch.from_numpy(np.ascontiguousarray(s[k])).cuda()
        if case["kind"] != "noalloc":
            s["matrix"] = torch.from_numpy(np.ascontiguousarray(s["matrix"])).cuda()
    if case["kind"] == "noalloc":
        s["cells"] = torch.zeros((case["pairs"], 5), dtype=torch.int32, device="cuda")
    if "params" in s:
        # a ranker's weights live in a context of their own
        s["ctx"] = cm.Context(0)
        s["ctx"].ranker_set_params(s["params"])
    else:
        s["ctx"] = cm.default_context()
    if case["kind"] == "allpairs":
        rows = 64 * case["proteins"]
        if case["device"]:
            s["found"] = (torch.zeros((rows, 2), dtype=torch.int32, device="cuda"),
                          torch.zeros(rows, dtype=torch.int32, device="cuda"))
        else:
            s["found"] = np.zeros((rows, 2), np.int32), np.zeros(rows, np.int32)
    return s


def run(state):
    s = state
    case, ctx, kind = s["case"], s["ctx"], s["case"]["kind"]
    if kind in ("search", "pairs", "long"):
        return ctx.sw_score_batch(s["seqs"], s["offsets"], s["pairs"], s["matrix"], GAP_OPEN,
                                  GAP_EXTEND)
    if kind == "allpairs":
        p, _ = ctx.sw_allpairs(s["seqs"], s["offsets"], s["matrix"], GAP_OPEN, GAP_EXTEND,
                               T_PAM if case["alphabet"] == 24 else T, part=case["parts"] // 3,
                               n_parts=case["parts"], flags=cm.CM_ASCII if case["ascii"] else 0,
                               pairs_out=s["found"][0], scores_out=s["found"][1])
        return len(p), s["found"][0], s["found"][1]
    if kind == "cells":
        return ctx.sw_cells_batch(s["seqs"], s["offsets"], s["pairs"], s["matrix"], GAP_OPEN,
                                  GAP_EXTEND)
    if kind == "noalloc":
        return cm.sw_cells_batch_noalloc(s["seqs"], s["offsets"], s["pairs"], s["matrix"],
                                         GAP_OPEN, GAP_EXTEND, s["cells"])
    if kind == "align":
        cells, offs, runs = ctx.sw_align_batch(s["seqs"], s["offsets"], s["pairs"], s["matrix"],
                                               GAP_OPEN, GAP_EXTEND)
        return cells, offs, _padded(runs, _ALIGN_RUNS * case["pairs"])
    if kind == "embed":
        if case["pairs"]:
            return ctx.ranker_logits(s["seqs"], s["offsets"], s["pairs"])
        return ctx.ranker_embed(s["seqs"], s["offsets"])
    if kind == "grad":
        return ctx.ranker_loss_grad(s["seqs"], s["offsets"], s["pairs"], s["labels"])
    if kind == "train":
        ctx.ranker_set_params(s["params"])         # every pass trains from the same weights
        loss = ctx.ranker_train(s["seqs"], s["offsets"], s["pairs"], s["labels"], epochs=1,
                                batch_pairs=15 * case["group"] + 64, lr=1e-3, seed=13,
                                flags=cm.CM_TRAIN_COMPONENTS | cm.CM_TRAIN_COSINE)
        return loss, ctx.ranker_get_params()
    t, mt = (T_PAM, M_T_PAM) if case["alphabet"] == 24 else (T, M_T)
    if case["mode"] == "greedy":
        r = ctx.greedy_cluster(s["seqs"], s["offsets"], s["matrix"], GAP_OPEN, GAP_EXTEND, t, mt,
                               M_U)
    else:
        r = ctx.cluster_merge(s["seqs"], s["offsets"], s["matrix"], GAP_OPEN, GAP_EXTEND, t, mt,
                              M_U, merge_mode=cm.CM_MERGE_PARTIAL if case["mode"] == "partial"
                              else cm.CM_MERGE_SEQUENTIAL)
    reps = np.array([c[0] for c in r["clusters"]], np.int32)
    sizes = np.array([len(c[1]) for c in r["clusters"]], np.int64)
    members = np.array([m for c in r["clusters"] for m in c[1]], np.int32)
    n = case["proteins"]
    return (_padded(reps, n), _padded(sizes, n), _padded(members, 16 * n),
            _padded(r["pairs"], 64 * n))


# ---- what a pass cannot do without ------------------------------------------------------------
CELL_OPS = 7                           # E 2, F 2, H 2, running maximum 1
EMBED_FLOPS = 2 * 9 * 128 * (32 + 128 + 128)      # per residue, forward


def work(case):
    kind = case["kind"]
    s = _inputs(case, 1)
    lens = np.diff(s["offsets"]).astype(np.float64)
    bytes_ = float(len(s["seqs"]) + 8 * len(s["offsets"]))
    if "pairs" in s:
        bytes_ += 8.0 * len(s["pairs"])
    if kind in ("search", "pairs", "long", "cells", "noalloc", "align"):
        cells = float((lens[s["pairs"][:, 0]] * lens[s["pairs"][:, 1]]).sum())
        # the start cell needs a second, reversed matrix; a traceback walks one path
        both = 1 if kind in ("search", "pairs", "long") else 2
        bytes_ += len(s["pairs"]) * (4.0 if both == 1 else 20.0)
        return {"bytes": bytes_, "flops": CELL_OPS * cells * both}
    if kind in ("allpairs", "cluster"):
        # a clustering compares a part of all pairs: counted whole, as its upper bound
        cells = (lens.sum() ** 2 - (lens ** 2).sum()) / 2 / case.get("parts", 1)
        return {"bytes": bytes_, "flops": CELL_OPS * cells}
    weights = 4.0 * len(s["params"])
    if kind == "embed":
        used = lens if not case["pairs"] else lens[np.unique(s["pairs"])]
        return {"bytes": bytes_ + weights / 2 + (4.0 * case["pairs"] or 512.0 * len(lens)),
                "flops": EMBED_FLOPS * float(used.sum())}
    rows = float(lens[np.unique(s["pairs"])].sum())
    return {"bytes": bytes_ + 2 * weights + 4.0 * len(s["labels"]), "flops": 3 * EMBED_FLOPS * rows}


# ---- the same results in 64 bits --------------------------------------------------------------
def _scores64(s, pairs, matrix):
    """Affine-gap local alignment scores, int64, row by row over many pairs at once: within a
    row E(j) = max over k < j of H(k) - open - (j - k - 1) * extend, a running maximum."""
    dev = _DEVICE
    off = torch.from_numpy(s["offsets"]).to(dev)
    seqs = torch.from_numpy(s["seqs"].astype(np.int64)).to(dev)
    mat = torch.from_numpy(np.asarray(matrix).astype(np.int64)).to(dev)
    p = torch.from_numpy(pairs.astype(np.int64)).to(dev)
    m, n = off[p[:, 0] + 1] - off[p[:, 0]], off[p[:, 1] + 1] - off[p[:, 1]]
    out = torch.zeros(len(p), dtype=torch.int64, device=dev)
    order = torch.argsort(m * 8192 + n)
    for part in torch.split(order, 4096):
        mm, nn = m[part], n[part]
        rows, cols = int(mm.max()), int(nn.max())
        j = torch.arange(cols, device=dev)
        inside = j[None, :] < nn[:, None]
        b = seqs[(off[p[part, 1]][:, None] + j[None, :]).clamp(max=len(seqs) - 1)]
        h = torch.zeros((len(part), cols + 1), dtype=torch.int64, device=dev)
        f = torch.full((len(part), cols), -(1 << 40), dtype=torch.int64, device=dev)
        best = torch.zeros(len(part), dtype=torch.int64, device=dev)
        for i in range(rows):
            a = seqs[(off[p[part, 0]] + i).clamp(max=len(seqs) - 1)]
            f = torch.maximum(f - GAP_EXTEND, h[:, 1:] - GAP_OPEN)
            d = torch.maximum(h[:, :-1] + mat[a[:, None], b], f).clamp(min=0)
            run_max = torch.cummax(d + GAP_EXTEND * j, dim=1).values
            e = torch.full_like(d, -(1 << 40))
            e[:, 1:] = run_max[:, :-1] - GAP_OPEN - GAP_EXTEND * (j[1:] - 1)
            live = inside & (mm > i)[:, None]
            h[:, 1:] = torch.where(live, torch.maximum(d, e), torch.zeros_like(d))
            best = torch.maximum(best, h.max(dim=1).values)
        out[part] = best
    return out.cpu()


def _forward64(s, params, ids):
    """Pooled vectors of the sequences `ids` (float64), differentiable in `params`."""
    shapes = [(20, 32), (9, 32, 128), (128,), (9, 128, 128), (128,), (9, 128, 128), (128,), (), ()]
    w, o = [], 0
    for shp in shapes:
        k = int(np.prod(shp)) if shp else 1
        w.append(params[o:o + k].reshape(shp))
        o += k
    lens = np.diff(s["offsets"])[ids]
    first = np.cumsum(lens + 4) - lens                 # four zero rows before each sequence
    rows = int(first[-1] + lens[-1] + 4)
    seq_of = np.full(rows, -1)
    codes = np.zeros(rows, np.int64)
    at = np.repeat(first, lens) + np.arange(lens.sum()) - np.repeat(np.cumsum(lens) - lens, lens)
    seq_of[at] = np.repeat(np.arange(len(ids)), lens)
    codes[at] = s["seqs"][np.repeat(s["offsets"][ids], lens) + np.arange(lens.sum()) -
                          np.repeat(np.cumsum(lens) - lens, lens)]
    dev = params.device
    at, codes = torch.from_numpy(at).to(dev), torch.from_numpy(codes).to(dev)
    real = torch.from_numpy((seq_of >= 0).astype(np.float64)).to(dev)[:, None]

    def conv(x, k, b):
        xp = torch.nn.functional.pad(x, (0, 0, 4, 4))
        y = sum(xp[t:t + rows] @ k[t] for t in range(9))
        return (y + b) * real

    z = torch.relu(conv(w[0][codes] * real, w[1], w[2]))
    z = torch.relu(conv(z, w[3], w[4]))
    z = conv(z, w[5], w[6])
    v = torch.zeros((len(ids), 128), dtype=torch.float64, device=dev)
    v = v.index_add(0, torch.from_numpy(seq_of[seq_of >= 0]).to(dev), z[at])
    return v / torch.from_numpy(lens.astype(np.float64)).to(dev)[:, None], w[7], w[8]


def _logits64(v, alpha, beta, a, b):
    va, vb = v[a], v[b]
    den = ((va * va).sum(1) + 1e-6) * ((vb * vb).sum(1) + 1e-6)
    return alpha * (va * vb).sum(1) / den.sqrt() + beta


def exact(case, seed):
    kind = case["kind"]
    s = _inputs(case, seed)
    if kind == "search" or (kind == "pairs" and case["pairs"] <= 10000):
        return _scores64(s, s["pairs"], _matrix(case))
    if kind == "embed":
        p = torch.from_numpy(s["params"].astype(np.float64)).to(_DEVICE)
        v, alpha, beta = [], None, None
        for ids in np.array_split(np.arange(case["proteins"]), -(-case["proteins"] // 500)):
            x, alpha, beta = _forward64(s, p, ids)
            v.append(x)
        v = torch.cat(v)
        if not case["pairs"]:
            return v.cpu()
        i = torch.from_numpy(s["pairs"].astype(np.int64)).to(_DEVICE)
        return _logits64(v, alpha, beta, i[:, 0], i[:, 1]).cpu()
    if kind == "grad":
        p = torch.from_numpy(s["params"].astype(np.float64)).to(_DEVICE).requires_grad_()
        ids, inv = np.unique(s["pairs"], return_inverse=True)
        v, alpha, beta = _forward64(s, p, ids)
        i = torch.from_numpy(inv.reshape(-1, 2).astype(np.int64)).to(_DEVICE)
        z = _logits64(v, alpha, beta, i[:, 0], i[:, 1])
        y = torch.from_numpy(s["labels"].astype(np.float64)).to(_DEVICE)
        loss = torch.nn.functional.binary_cross_entropy_with_logits(z, y)
        loss.backward()
        return loss.detach().cpu(), p.grad.cpu()
    return None                            # whole numbers, or the course of a training run
