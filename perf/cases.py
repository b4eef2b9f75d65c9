"""The measured workloads: what a user of this library has it do.

A case is one call of a public entry point on a text and a compiled pattern
set, with everything a program would hold between calls (the compiled set,
the workspace, the result buffers) made by :func:`prepare`. The texts have the
shapes of this repository's own workloads: EST-shaped nucleotides (sequences
of lognormal length separated by newlines, about 1 % ``N``), i.i.d. ACGT, and
protein-like text over 20 letters for the general-alphabet path. Half of each
pattern set is copied from the text, half is drawn at random.

Whole numbers come back everywhere: per-pattern counts, the total, and the
sorted ``(position << 32) | pattern`` keys.
"""
from __future__ import annotations

import numpy as np
import torch

from paper_1407_2889_gb300 import pmscan as pm

MIB = 1 << 20
DNA = b"ACGT"
PROTEIN = b"ACDEFGHIKLMNPQRSTVWY"

# ---------------------------------------------------------------------------
# The listed cases
# ---------------------------------------------------------------------------
# entry:    "device" pm_scan_device, "host" pm_scan_to_host, "batch" the
#           batched scan
# algo:     how the set is compiled
# text:     "est", "uniform" (ACGT without separators) or "protein"
# n, d:     text bytes and patterns; lengths are uniform in [m_lo, m_hi]
# list:     the sorted occurrence list too, or counts only


def _scan(name, algo, text, n, d, m_lo, m_hi=0, list_=True, entry="device", B=0):
    return {"name": name, "entry": entry, "algo": algo, "text": text, "n": n, "d": d,
            "m_lo": m_lo, "m_hi": m_hi or m_lo, "list": list_, "B": B, "k": 1}


def listed():
    return [
        # a short interactive query: launches and latency count
        _scan("ac_small_1mib", "ac", "uniform", MIB, 100, 8),
        # the headline scan: a whole EST snapshot against many short tags,
        # every occurrence listed (about one position in nine matches)
        _scan("ac_est_1gib_d8000_m8", "ac", "est", 1024 * MIB, 8000, 8),
        # a census: per-pattern counts of 16-mers, no list
        _scan("ac_est_counts_d1000_m16", "ac", "est", 256 * MIB, 1000, 16, list_=False),
        # read-length probes, the largest table of the evaluation sets
        _scan("ac_est_d20000_m32", "ac", "est", 256 * MIB, 20000, 32),
        # a dictionary far larger than on-chip memory
        _scan("ac_est_d100000_m32", "ac", "est", 256 * MIB, 100000, 32),
        # an alphabet without the nucleotide shortcut, odd text length
        _scan("ac_protein_d2000_m12", "ac", "protein", 64 * MIB + 4321, 2000, 12),
        # Wu-Manber with 3-character blocks
        _scan("wm_est_d8000_m16", "wm", "est", 256 * MIB, 8000, 16, B=3),
        # failure-less automaton on a small set of short patterns
        _scan("pfac_est_d1000_m8", "pfac", "est", 128 * MIB, 1000, 8),
        # patterns of their own lengths, both methods
        _scan("acv_est_d8000_m8_16", "acv", "est", 256 * MIB, 8000, 8, 16),
        _scan("wmv_est_d1000_m8_16", "wmv", "est", 128 * MIB + 77, 1000, 8, 16, B=3),
        # many independent small texts, each against its own set, in one launch
        {"name": "batch_1024", "entry": "batch", "algo": "ac", "text": "est", "n": 1 << 22, "d": 10000,
         "m_lo": 8, "m_hi": 64, "list": True, "B": 0, "k": 1024},
        # a host text scanned end to end: copies in and out included
        _scan("host_est_256mib_d8000_m8", "ac", "est", 256 * MIB, 8000, 8, entry="host"),
    ]


def _log_uniform(rng, lo, hi):
    return int(min(hi, max(lo, round(lo * (hi / lo) ** rng.random()))))


def draw(rng):
    kind = rng.choice(["ac", "ac", "ac_counts", "ac_long", "protein", "wm", "pfac", "acv", "wmv", "batch", "host"])
    if kind == "batch":
        case = {"entry": "batch", "algo": "ac", "text": "est", "n": 1 << 22, "d": 10000, "m_lo": 8,
                "m_hi": 64, "list": rng.random() < 0.75, "B": 0, "k": _log_uniform(rng, 64, 1024)}
        return case
    if kind in ("ac", "ac_counts", "host"):
        n, d, m = _log_uniform(rng, MIB // 16, 256 * MIB), _log_uniform(rng, 100, 20000), rng.randint(8, 32)
        case = _scan("", "ac", rng.choice(["est", "uniform"]), n, d, m, list_=kind != "ac_counts",
                     entry="host" if kind == "host" else "device")
    elif kind == "ac_long":  # long patterns, large sets
        m = rng.randint(24, 64)
        case = _scan("", "ac", "est", _log_uniform(rng, MIB, 256 * MIB), _log_uniform(rng, 100, 100000), m,
                     list_=rng.random() < 0.5)
    elif kind == "protein":
        case = _scan("", rng.choice(["ac", "ac", "wm"]), "protein", _log_uniform(rng, MIB // 16, 64 * MIB),
                     _log_uniform(rng, 100, 5000), rng.randint(6, 24), list_=rng.random() < 0.75, B=2)
    elif kind in ("wm", "pfac"):
        case = _scan("", kind, "est", _log_uniform(rng, MIB // 16, 64 * MIB), _log_uniform(rng, 100, 20000),
                     rng.randint(8, 32), list_=rng.random() < 0.75, B=rng.randint(2, 3))
    else:
        lo = rng.randint(8, 16)
        case = _scan("", kind, "est", _log_uniform(rng, MIB // 16, 64 * MIB), _log_uniform(rng, 100, 8000),
                     lo, lo + rng.randint(1, 16), list_=rng.random() < 0.75, B=rng.randint(2, 3))
    del case["name"]
    return case


def _expected_occ(n, d, m_lo, m_hi, kind):
    letters = 20.0 if kind == "protein" else 4.0
    clean = 0.988 if kind == "est" else 1.0
    per = 1.0 / (m_hi - m_lo + 1)
    return d // 2 + sum(per * n * d * (clean / letters) ** m for m in range(m_lo, m_hi + 1))


def _capacity(n, d, m_lo, m_hi, kind):
    """Room for the list: a quarter more than expected. What a scan leaves
    unused stays zero."""
    return int(1.25 * _expected_occ(n, d, m_lo, m_hi, kind)) + d + 1024


# ---------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------
def _device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _text(kind, n, seed):
    """n bytes of text on the device, from the seed alone."""
    dev = _device()
    g = torch.Generator(device=dev)
    g.manual_seed(seed * 1000003 + 17)
    alpha = torch.tensor(list(PROTEIN if kind == "protein" else DNA), dtype=torch.uint8, device=dev)
    out = torch.empty(n, dtype=torch.uint8, device=dev)
    step = 64 * MIB
    for a in range(0, n, step):
        b = min(n, a + step)
        v = torch.randint(0, 1 << 24, (b - a,), dtype=torch.int32, device=dev, generator=g)
        piece = alpha[(v % len(alpha)).long()]
        if kind == "est":
            piece[torch.randint(0, 16384, (b - a,), dtype=torch.int32, device=dev, generator=g) < 164] = ord("N")
        out[a:b] = piece
    if kind != "uniform":  # a newline after each sequence
        rng = np.random.default_rng(seed * 7919 + 5)
        z = rng.standard_normal(n // 100 + 16)
        lens = np.clip(np.rint(450.0 * np.exp(0.6 * z)), 100, 1200).astype(np.int64)
        sep = np.cumsum(lens + 1) - 1
        out[torch.from_numpy(sep[sep < n]).to(dev)] = ord("\n")
    return out


def _patterns(text, kind, d, m_lo, m_hi, seed):
    """d byte strings (int64 lengths, (d, m_hi) uint8 rows padded with 0): the
    half of them windows of the text without separators or unknown letters, the
    rest i.i.d., in random order."""
    rng = np.random.default_rng(seed * 104729 + 11)
    alpha = np.frombuffer(PROTEIN if kind == "protein" else DNA, dtype=np.uint8)
    lens = rng.integers(m_lo, m_hi + 1, d)
    rows = alpha[rng.integers(0, alpha.size, (d, m_hi))]
    n = int(text.numel())
    ok = torch.zeros(256, dtype=torch.bool, device=text.device)
    ok[torch.from_numpy(alpha.astype(np.int64)).to(text.device)] = True
    got, want, tries = 0, d // 2, 0
    span = torch.arange(m_hi, device=text.device)
    while got < want and n >= m_hi and tries < 20:
        tries += 1
        starts = torch.from_numpy(rng.integers(0, n - m_hi + 1, 2 * (want - got) + 64)).to(text.device)
        win = text[starts[:, None] + span[None, :]]
        win = win[ok[win.long()].all(dim=1)][: want - got].cpu().numpy()
        rows[got:got + len(win)] = win
        got += len(win)
    rows = rows[rng.permutation(d)]
    rows[np.arange(m_hi)[None, :] >= lens[:, None]] = 0
    return lens, np.ascontiguousarray(rows)


def _compile(case, lens, rows):
    algo = case["algo"]
    if algo in ("ac", "wm", "pfac"):
        if algo == "ac":
            return pm.PatternSet.ac(rows)
        return pm.PatternSet.pfac(rows) if algo == "pfac" else pm.PatternSet.wm(rows, case["B"])
    off = np.zeros(lens.size + 1, np.int64)
    np.cumsum(lens, out=off[1:])
    cat = rows[np.arange(rows.shape[1])[None, :] < lens[:, None]]
    return pm.PatternSet.acv((cat, off)) if algo == "acv" else pm.PatternSet.wmv((cat, off), case["B"])


def _batch_plan(case):
    """(offset, length, d, m) of each instance: lengths log-uniform from 1 KiB
    to n, sets log-uniform from 10 to d patterns, slices of one EST text. The
    shapes belong to the case; a seed fills them."""
    rng = np.random.default_rng(15485863 + case["k"])
    base = 64 * MIB
    out = []
    for _ in range(case["k"]):
        u = rng.random(4)
        ln = int(round(1024 * (case["n"] / 1024) ** u[0]))
        d = int(round(10 * (case["d"] / 10) ** u[2]))
        m = case["m_lo"] + int(u[3] * (case["m_hi"] - case["m_lo"] + 1))
        out.append((int(u[1] * (base - ln)) // 16 * 16, ln, d, m))
    return base, out


def _batch_patterns(base_host, plan, j, seed):
    """Instance j's patterns from at least 64 KiB of text at its slice."""
    off, ln, d, m = plan[j]
    lo = max(0, min(off, base_host.numel() - max(ln, 1 << 16)))
    return _patterns(base_host[lo:lo + max(ln, 1 << 16)], "est", d, m, m, seed * 65537 + j)[1]


def prepare(case, seed):
    state = {"case": case, "flags": 0 if case["list"] else pm.PM_COUNTS_ONLY}
    if case["entry"] == "batch":
        base, plan = _batch_plan(case)
        text = _text("est", base, seed)
        host = text.cpu()
        sets = [pm.PatternSet.ac(_batch_patterns(host, plan, j, seed)) for j in range(case["k"])]
        offs, lens = [p[0] for p in plan], [p[1] for p in plan]
        caps = [_capacity(ln, d, m, m, "est") for _, ln, d, m in plan]
        b = pm.Batch(sets, text, offs, lens, caps if case["list"] else None)
        b.occ.zero_()
        state.update(batch=b)
        return state
    text = _text(case["text"], case["n"], seed)
    lens, rows = _patterns(text, case["text"], case["d"], case["m_lo"], case["m_hi"], seed)
    s = _compile(case, lens, rows)
    cap = _capacity(case["n"], case["d"], case["m_lo"], case["m_hi"], case["text"])
    state.update(set=s)
    if case["entry"] == "host":
        pin = torch.cuda.is_available()
        state.update(text=text.cpu().pin_memory() if pin else text.cpu(),
                     counts=torch.zeros(case["d"], dtype=torch.int64, pin_memory=pin),
                     occ=torch.zeros(cap, dtype=torch.int64, pin_memory=pin))
        return state
    dev = text.device
    ws = s.workspace_bytes(case["n"], counts_only=not case["list"])
    state.update(text=text, counts=torch.zeros(case["d"], dtype=torch.int64, device=dev),
                 occ=torch.zeros(cap if case["list"] else 1, dtype=torch.int64, device=dev), cap=cap,
                 n_occ=torch.zeros(1, dtype=torch.int64, device=dev), ws_bytes=ws,
                 ws=torch.empty(max(256, ws), dtype=torch.uint8, device=dev))
    return state


def run(state):
    case = state["case"]
    if case["entry"] == "batch":
        b = state["batch"]
        b.scan(torch.cuda.current_stream())
        out = {"counts": b.counts, "n_occ": b.n_occ}
        if case["list"]:
            out["occ"] = b.occ
        return out
    if case["entry"] == "host":
        total = pm.pm_scan_to_host(state["set"].h, state["text"], state["counts"], state["occ"], state["flags"],
                                   torch.cuda.current_stream())
        return {"counts": state["counts"], "n_occ": total, "occ": state["occ"]}
    pm.pm_scan_device(state["set"].h, state["text"], case["n"], state["flags"], state["counts"],
                      state["occ"] if case["list"] else None, state["cap"], state["n_occ"], state["ws"],
                      state["ws_bytes"], torch.cuda.current_stream())
    out = {"counts": state["counts"], "n_occ": state["n_occ"]}
    if case["list"]:
        out["occ"] = state["occ"]
    return out


# ---------------------------------------------------------------------------
# What a pass cannot do without
# ---------------------------------------------------------------------------
def work(case):
    """The text read once, the counts and the keys written once; integer work
    only, no floating-point operations."""
    if case["entry"] == "batch":
        total = 0.0
        for _, ln, d, m in _batch_plan(case)[1]:
            total += ln + 8 * d + 8 + (8 * _expected_occ(ln, d, m, m, "est") if case["list"] else 0)
        return {"bytes": total, "flops": 0.0}
    total = case["n"] + 8 * case["d"] + 8
    if case["list"]:
        total += 8 * _expected_occ(case["n"], case["d"], case["m_lo"], case["m_hi"], case["text"])
    return {"bytes": float(total), "flops": 0.0}


# ---------------------------------------------------------------------------
# The definition, in plain torch: every (i, r) with text[i : i + len_r] = p^r
# ---------------------------------------------------------------------------
def _occurrences(text, lens, rows, kind):
    """(sorted keys, counts): a window's first k letters as one integer, looked
    up in the sorted patterns; the candidates compared letter by letter."""
    dev = text.device
    letters = PROTEIN if kind == "protein" else DNA
    bits = 5 if kind == "protein" else 2
    n, d = int(text.numel()), len(lens)
    m_lo, m_hi = int(lens.min()), int(lens.max())
    k = min(m_lo, 62 // bits)
    cls = torch.full((256,), -1, dtype=torch.int64, device=dev)
    for c, b in enumerate(letters):
        cls[b] = c
    P = torch.from_numpy(rows).to(dev)
    L = torch.from_numpy(lens.astype(np.int64)).to(dev)
    pk = torch.zeros(d, dtype=torch.int64, device=dev)
    for j in range(k):
        pk = (pk << bits) | cls[P[:, j].long()]
    pk, order = torch.sort(pk, stable=True)
    uniq, mult = torch.unique_consecutive(pk, return_counts=True)
    first = torch.cumsum(mult, 0) - mult
    found = []
    step = 64 * MIB
    for a in range(0, max(0, n - m_lo + 1), step):
        b = min(n - m_lo + 1, a + step)
        code = torch.zeros(b - a, dtype=torch.int64, device=dev)
        good = torch.ones(b - a, dtype=torch.bool, device=dev)
        for j in range(k):
            c = cls[text[a + j:b + j].long()]
            good &= c >= 0
            code = (code << bits) | (c & ((1 << bits) - 1))
        at = torch.searchsorted(uniq, code).clamp_(max=uniq.numel() - 1)
        pos = torch.nonzero((uniq[at] == code) & good).flatten()
        at = at[pos]
        rep = mult[at]
        pos_r = torch.repeat_interleave(pos, rep) + a
        inner = torch.arange(pos_r.numel(), device=dev) - torch.repeat_interleave(torch.cumsum(rep, 0) - rep, rep)
        r = order[torch.repeat_interleave(first[at], rep) + inner]
        alive = pos_r + L[r] <= n
        for j in range(k, m_hi):
            t = text[(pos_r + j).clamp_(max=n - 1)]
            alive &= (j >= L[r]) | (t == P[r, j])
        found.append((pos_r[alive] << 32) | r[alive])
    keys = torch.sort(torch.cat(found))[0] if found else torch.zeros(0, dtype=torch.int64, device=dev)
    return keys, torch.bincount(keys & 0xFFFFFFFF, minlength=d)


def _padded(keys, cap):
    out = torch.zeros(cap, dtype=torch.int64, device=keys.device)
    out[: min(cap, keys.numel())] = keys[:cap]
    return out


def exact(case, seed):
    if case["entry"] == "batch":
        base, plan = _batch_plan(case)
        text = _text("est", base, seed)
        host = text.cpu()
        keys, counts = [], []
        for j, (off, ln, d, m) in enumerate(plan):
            rows = _batch_patterns(host, plan, j, seed)
            kk, cc = _occurrences(text[off:off + ln], np.full(d, m, np.int64), rows, "est")
            keys.append(kk)
            counts.append(cc)
        n_occ = torch.tensor([kk.numel() for kk in keys], dtype=torch.int64, device=text.device)
        out = {"counts": torch.cat(counts), "n_occ": n_occ}
        if case["list"]:
            out["occ"] = torch.cat([_padded(kk, _capacity(ln, d, m, m, "est"))
                                    for kk, (_, ln, d, m) in zip(keys, plan)])
        return out
    text = _text(case["text"], case["n"], seed)
    lens, rows = _patterns(text, case["text"], case["d"], case["m_lo"], case["m_hi"], seed)
    keys, counts = _occurrences(text, lens, rows, case["text"])
    total = int(keys.numel())
    keys = _padded(keys, _capacity(case["n"], case["d"], case["m_lo"], case["m_hi"], case["text"]))
    if case["entry"] == "host":
        return {"counts": counts.cpu(), "n_occ": total, "occ": keys.cpu()}
    out = {"counts": counts, "n_occ": torch.tensor([total], dtype=torch.int64, device=text.device)}
    if case["list"]:
        out["occ"] = keys
    return out
