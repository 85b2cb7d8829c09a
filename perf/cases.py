"""Workloads that measure the sparse-state library as its users run it.

A case is one simulation from |0...0> through the Python binding (reset, the
gates one call each, the readout a program would make), a graph replay of one,
or a readout of a loaded state.  The circuits are the seeded synthetic ones of
workloads.py and qlss.py at the sizes of this repository's benchmark and tests
and at sizes between them; every family is drawn over its whole range, odd
register widths, one- and two-word keys and both amplitude types among them.

Outputs: the exported state (keys ascending, amplitudes), or what a program
reads of it instead where it holds millions of branches or a number of them
that depends on the data: marginal probabilities, the norm, the system
vector of a walk.  An exported state whose size depends on the data is padded
to the circuit's bound.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2503_15118_gb300 import qlss, sqs
from paper_2503_15118_gb300 import workloads as W


def listed():
    return [
        # The smallest real use: one 20-qubit circuit (three registers, a QRAM
        # load, 200 mixed gates, at most 4096 branches) issued gate by gate and
        # read out whole.  Launches and host calls are what it costs.
        {"name": "circuit20", "family": "circuit20", "cap": 4096, "gates": 200, "graph": False,
         "fp32": False},
        # The same circuit captured once and replayed, as a program that runs
        # one circuit many times does.
        {"name": "circuit20_graph", "family": "circuit20", "cap": 4096, "gates": 200,
         "graph": True, "fp32": False},
        # Thousands of such circuits batched in one state, each with its own
        # table: throughput of long runs of mixed gates on a large state.
        {"name": "circuit20_batch", "family": "batch20", "cap": 4096, "gates": 200,
         "inst_bits": 12, "fp32": False},
        # The benchmark's workload: a 64-qubit random circuit, 24 branching
        # gates among 500 others, 2^24 branches at its peak.
        {"name": "random64", "family": "random", "widths": "16,16,16,16", "branch": 24,
         "perm": 500, "cancel": 8, "fp32": False},
        # An ordinary size of it, registers of odd widths, FP32 storage.
        {"name": "random59_fp32", "family": "random", "widths": "13,19,10,17", "branch": 19,
         "perm": 233, "cancel": 5, "fp32": True},
        # QRAM rounds on two-word keys (load, add into an accumulator, rotate
        # the loaded data and back, unload), the benchmark's table size.
        {"name": "qram84", "family": "qram", "addr": 20, "rounds": 3, "ry": 4, "fp32": False},
        # The same over a small odd table, FP32 storage.
        {"name": "qram77_fp32", "family": "qram", "addr": 13, "rounds": 5, "ry": 3, "fp32": True},
        # The linear-system walk at the benchmark's matrix size, one step in
        # the middle of the schedule.
        {"name": "walk1024", "family": "walk", "n": 10, "half_band": 8, "kappa": 10.0, "steps": 1,
         "nonherm": False, "fp32": False},
        # A small non-Hermitian system, several steps.
        {"name": "walk128_nonherm", "family": "walk", "n": 7, "half_band": 5, "kappa": 50.0,
         "steps": 3, "nonherm": True, "fp32": False},
        # Many small systems walked at once in one state (two-word keys).
        {"name": "walk_batch", "family": "walk_batch", "inst": 64, "n_max": 7, "steps": 2,
         "fp32": False},
        # Arithmetic oracles, general and controlled single-qubit matrices,
        # swaps and phases on two-word keys.
        {"name": "arith101", "family": "arith", "widths": "24,31,24,14", "spread": 20, "gates": 90,
         "branch": 6, "fp32": False},
        # Reading a large loaded state: marginals of a narrow and of a 40-bit register.
        {"name": "readout", "family": "readout", "widths": "12,40,35", "count": 3000017,
         "fp32": False},
    ]


def _log2_between(rng, lo, hi):
    return lo + (hi - lo) * rng.random()


def draw(rng):
    """One more case of the same ranges (spread over the logarithm of the work)."""
    f = rng.choice(["circuit20", "batch20", "random", "random", "qram", "walk", "walk_batch",
                    "arith", "readout"])
    fp32 = rng.random() < 0.35
    if f == "circuit20":
        return {"family": f, "cap": int(2 ** _log2_between(rng, 9, 13.4)),
                "gates": rng.randint(60, 260), "graph": rng.random() < 0.4, "fp32": fp32}
    if f == "batch20":
        bits = rng.randint(5, 12)
        return {"family": f, "cap": int(2 ** _log2_between(rng, 10, 12)),
                "gates": rng.randint(60, 220), "inst_bits": bits, "fp32": fp32}
    if f == "random":
        branch = rng.randint(13, 24)
        widths = [rng.randint(9, 16) for _ in range(4)]
        if rng.random() < 0.3:  # two-word keys
            widths = [rng.randint(17, 30) for _ in range(4)]
            branch = min(branch, 22)
        return {"family": f, "widths": ",".join(map(str, widths)), "branch": branch,
                "perm": rng.randint(60, 500), "cancel": rng.randint(2, 8), "fp32": fp32}
    if f == "qram":
        addr = rng.randint(10, 19)
        return {"family": f, "addr": addr, "rounds": rng.randint(1, 4), "ry": rng.randint(2, 5),
                "fp32": fp32}
    if f == "walk":
        n = rng.randint(5, 9)
        return {"family": f, "n": n, "half_band": rng.randint(1, min(12, (1 << n) // 4)),
                "kappa": float(rng.choice([10, 50, 100])), "steps": rng.randint(1, 3),
                "nonherm": rng.random() < 0.4, "fp32": fp32}
    if f == "walk_batch":
        return {"family": f, "inst": rng.choice([16, 32, 64, 100]), "n_max": rng.randint(4, 7),
                "steps": rng.randint(1, 2), "fp32": fp32}
    if f == "arith":
        w = rng.randint(18, 26)
        widths = [w, rng.randint(20, 36), w, rng.randint(5, 15)]
        return {"family": f, "widths": ",".join(map(str, widths)),
                "spread": rng.randint(12, 20), "gates": rng.randint(30, 120),
                "branch": rng.randint(2, 6), "fp32": fp32}
    widths = [rng.randint(6, 14), rng.randint(24, 48), rng.randint(23, 40)]
    return {"family": f, "widths": ",".join(map(str, widths)),
            "count": int(2 ** _log2_between(rng, 12, 22.5)), "fp32": fp32}


# ---- the circuits -----------------------------------------------------------------

def _widths(case):
    return [int(w) for w in case["widths"].split(",")]


def _capped_gates(seed, n_gates, cap):
    """The 20-qubit circuit: H on the address bits, a QRAM load, then seeded
    gates of six kinds, each kept when the keys that can be reached stay at
    most `cap` (counted on the key set, without amplitudes).  Returns the
    circuit and the reachable keys before every gate."""
    circ, rng = W.config1_prefix(seed)
    off = np.cumsum([0] + circ["widths"])
    table = circ["tables"][0].astype(np.int64)
    keys = np.arange(256, dtype=np.int64)
    keys = keys | (table[keys] << off[1])
    counts = [1 << b for b in range(8)] + [256]
    gates = circ["gates"]

    def met(ctrls):
        on = np.ones(keys.shape, bool)
        for r, b, v in ctrls:
            on &= ((keys >> int(off[r] + b)) & 1) == v
        return on

    while len(gates) < 9 + n_gates:
        g = W.config1_candidates(rng)
        new = keys
        if g[0] == "x":
            new = np.where(met(g[3]), keys ^ (1 << int(off[g[1]] + g[2])), keys)
        elif g[0] in ("h", "ry"):
            t = 1 << int(off[g[1]] + g[2])
            new = np.union1d(keys, keys ^ t)
        if new.shape[0] > cap:
            continue
        counts.append(keys.shape[0])
        gates.append(g)
        keys = new
    return circ, counts


def _arith_circuit(case, seed):
    """H on `spread` qubits of the first two registers, then seeded arithmetic,
    swaps, phases and diagonal matrices with `branch` general, controlled or
    angle-register interference steps spread among them."""
    widths = _widths(case)
    rng = np.random.default_rng(seed)
    half = case["spread"] // 2
    lo = rng.choice(widths[0], size=half, replace=False)
    hi = rng.choice(widths[1], size=case["spread"] - half, replace=False)
    gates = [("h", 0, int(b), ()) for b in lo] + [("h", 1, int(b), ()) for b in hi]
    plain = ("muladd", "mulc", "divxor", "add", "sub", "swap", "cx", "ccx", "cphase", "diag",
             "adiag")
    qs = W._qubits(widths)
    at = set(np.linspace(2, case["gates"] - 1, case["branch"]).astype(int).tolist())
    for i in range(case["gates"]):
        if i in at:
            k = ("cu1q", "ch", "u1q", "cry")[int(rng.integers(4))]
            gates.append(W._draw_gate(rng, (k,), qs, widths, 0))
        else:
            gates.append(W._draw_gate(rng, plain, qs, widths, 0))
    return {"widths": widths, "eps": 1e-14, "tables": [], "gates": gates, "name": "arith"}


def _circuit(case, seed):
    f = case["family"]
    if f == "circuit20":
        return _capped_gates(seed, case["gates"], case["cap"])[0]
    if f == "batch20":
        stored = _capped_gates(seed, case["gates"], case["cap"])[0]
        return W.config1_batch(stored, inst_bits=case["inst_bits"], seed=seed)
    if f == "random":
        return W.config2(seed=seed, n_branch=case["branch"], n_perm=case["perm"],
                         n_cancel=case["cancel"], widths=_widths(case))
    if f == "qram":
        return W.config3(seed=seed, addr_bits=case["addr"], rounds=case["rounds"],
                         ry_bits=case["ry"])
    if f == "walk":
        make = qlss.config4_nonherm if case["nonherm"] else qlss.config4
        step = qlss.walk_step_nh if case["nonherm"] else qlss.walk_step
        cfg = make(seed=seed, N=1 << case["n"], half_band=case["half_band"], kappa=case["kappa"],
                   T=100)
        gates = list(cfg["prep"])
        for fs in cfg["steps"][50:50 + case["steps"]]:  # the middle of the schedule
            gates += step(cfg, fs)
        return {"widths": cfg["widths"], "eps": cfg["eps"], "tables": cfg["tables"],
                "gates": gates, "name": cfg["name"], "top": cfg["ids"]["TOP"],
                "bot": cfg["ids"]["BOT"],
                "system": [cfg["ids"][k] for k in ("TOP", "AH", "A1") if k in cfg["ids"]]}
    if f == "walk_batch":
        cfg = qlss.config5(seed=seed, n_inst=case["inst"], n_max=case["n_max"], T=100)
        c = qlss.batched_circuit(cfg, case["steps"])
        first = cfg["ids"]["STEP"]
        prep = len(qlss.batched_prep(cfg))
        # The middle of the schedule: the step counter starts at 50.
        c["gates"] = c["gates"][:prep] + [("add", first, -1, 50, ())] + c["gates"][prep:]
        c["top"], c["bot"] = cfg["ids"]["TOP"], cfg["ids"]["BOT"]
        c["inst"] = cfg["ids"]["INST"]
        return c
    if f == "arith":
        return _arith_circuit(case, seed)
    raise ValueError(f)


def _loaded(case, seed):
    """Distinct random keys and normalised complex amplitudes of a readout case.
    The first register's values are skewed (a few common ones), every value of
    the second occurs on two branches, the last register numbers the branches."""
    widths = _widths(case)
    n = case["count"]
    rng = np.random.default_rng(seed)
    r0 = (rng.random(n) ** 2 * (1 << widths[0])).astype(np.uint64)
    odd = np.uint64(rng.integers(0, 1 << 62) | 1)
    r1 = ((rng.permutation(n) >> 1).astype(np.uint64) * odd) & np.uint64((1 << widths[1]) - 1)
    r2 = rng.permutation(n).astype(np.uint64)
    off = np.cumsum([0] + widths)
    lo, hi = np.zeros(n, np.uint64), np.zeros(n, np.uint64)
    for r, o, w in zip((r0, r1, r2), off, widths):
        if o < 64:
            lo |= r << np.uint64(o)
            if o + w > 64:
                hi |= r >> np.uint64(64 - o)
        else:
            hi |= r << np.uint64(o - 64)
    a = rng.standard_normal((n, 2))
    a = a.view(np.complex128).reshape(-1)
    return lo, hi, a / math.sqrt(float(np.sum(np.abs(a) ** 2)))


# ---- a program's preparation and one pass -----------------------------------------

def prepare(case, seed):
    f = case["family"]
    if f == "readout":
        widths = _widths(case)
        st = sqs.State(widths, amp32=case["fp32"])
        st.import_(*_loaded(case, seed))
        return {"case": case, "st": st}
    circ = _circuit(case, seed)
    stream = torch.cuda.Stream()  # a side stream, which graph capture needs
    st = sqs.State(circ["widths"], amp32=case["fp32"], eps=circ["eps"],
                   stream=stream.cuda_stream)
    for t in circ["tables"]:
        st.table(t)
    state = {"case": case, "st": st, "circ": circ, "stream": stream}
    if case.get("graph"):
        state["graph"] = st.capture(circ, 4 * case["cap"])
    return state


def run(state):
    case, st = state["case"], state["st"]
    f = case["family"]
    if f == "readout":
        narrow, _ = st.probabilities(0)
        values, probs, norm = st.probabilities_sparse(1)
        return {"narrow": narrow, "values": values.view(np.int64), "probs": probs, "norm": norm}
    circ = state["circ"]
    if "graph" in state:
        state["graph"].launch()
    else:
        st.reset()
        st.run(circ)
    if f == "batch20":
        addr, norm = st.probabilities(0)
        inst, _ = st.probabilities(1)
        data, _ = st.probabilities(2)
        return {"addr": addr, "inst": inst, "data": data, "norm": norm}
    if f in ("walk", "walk_batch"):
        top, norm = st.probabilities(circ["top"])
        bot, _ = st.probabilities(circ["bot"])
        out = {"top": top, "bot": bot, "norm": norm}
        if "inst" in circ:
            out["inst"], _ = st.probabilities(circ["inst"])
        elif case["n"] <= 8:
            out["system"] = _system(circ, st.export())
        return out
    if f == "arith":
        narrow, norm = st.probabilities(3)
        return {"narrow": narrow, "norm": norm}
    out = _export(st)
    if f == "circuit20":
        return _padded(out, case["cap"])
    if f == "random":
        out["marginal"], out["norm"] = st.probabilities(0) if circ["widths"][0] <= 26 else \
            (None, st.probabilities(0, with_probs=False)[1])
        out = {k: v for k, v in out.items() if v is not None}
    return out


def _system(circ, state):
    """The walk's system vector: the amplitudes of |j>_TOP and the block qubits
    with every ancilla 0, over (block qubits, j); the solution is one block."""
    lo, hi, amps = state
    keys = lo.view(np.int64)
    off = np.cumsum([0] + circ["widths"])
    index = np.zeros(keys.shape, np.int64)
    used, place = 0, 0
    for r in circ["system"]:
        w = circ["widths"][r]
        index |= ((keys >> int(off[r])) & ((1 << w) - 1)) << place
        used |= ((1 << w) - 1) << int(off[r])
        place += w
    at = np.nonzero((keys & ~np.int64(used)) == 0)[0]
    v = np.zeros(1 << place, np.complex128)
    v[index[at]] = amps[at]
    return v


def _padded(state, size):
    """A state padded to `size` branches (the count itself is kept)."""
    n = state["lo"].shape[0]
    out = {"count": n}
    for k, v in state.items():
        out[k] = np.zeros(size, v.dtype)
        out[k][:n] = v
    return out


def _export(st):
    lo, hi, amps = st.export()
    return {"lo": lo.view(np.int64), "hi": hi.view(np.int64), "amps": amps}


# ---- what one pass cannot do without ----------------------------------------------

def work(case):
    """Bytes: every pass over the state that the circuit's structure needs --
    one per interference step on a fresh or mixed qubit (the branches in read,
    the branches out written), one per block of steps that stays inside the
    groups of one register -- plus the readout.  Flops: four real products and
    two sums per member and child of a step."""
    f = case["family"]
    amp = 8 if case["fp32"] else 16
    if f == "readout":
        rb = (8 if sum(_widths(case)) <= 64 else 16) + amp
        n = case["count"]
        return {"bytes": n * (2 * rb + 16), "flops": 6 * n}
    if f in ("circuit20", "batch20"):
        _, counts = _capped_gates(0, case["gates"], case["cap"])
        circ = _capped_gates(0, case["gates"], case["cap"])[0]
        scale = 1 << case.get("inst_bits", 0)
        counts = counts + [case["cap"]]
        moved = sum(counts[i] + counts[i + 1] for i, g in enumerate(circ["gates"])
                    if g[0] in ("h", "ry"))
        return {"bytes": scale * (moved + counts[-1]) * (8 + amp), "flops": 12 * scale * moved}
    if f == "random":
        rb = (8 if sum(_widths(case)) <= 64 else 16) + amp
        n = (1 << (case["branch"] + 1)) - 1            # sum of the inputs of the expansions
        m = 2 * n
        back = sum(3 << (case["branch"] - 1 - i) for i in range(case["cancel"]))
        return {"bytes": (n // 2 + m // 2 + back) * rb, "flops": 6 * (n + back)}
    if f == "qram":
        rb = 16 + amp
        n = 1 << case["addr"]
        steps = 2 * case["ry"] * (1 << case["ry"])
        return {"bytes": (3 * n + 2 * n * case["rounds"]) * rb + 4 * n * case["rounds"],
                "flops": 6 * n * steps * case["rounds"]}
    if f in ("walk", "walk_batch"):
        rb = (8 if f == "walk" else 16) + amp
        if f == "walk":
            n = 1 << (2 * case["n"] + (1 if case["nonherm"] else 0))
            blocks = 16 if not case["nonherm"] else 24
            levels = case["n"]
        else:
            n = case["inst"] << (2 * case["n_max"] - 3)
            blocks, levels = 16, case["n_max"]
        return {"bytes": n * rb * blocks * case["steps"],
                "flops": 6 * n * blocks * levels * case["steps"]}
    n = 1 << case["spread"]
    rb = 16 + amp
    return {"bytes": (2 * n + 3 * n * (1 << min(case["branch"], 2))) * rb,
            "flops": 12 * n * case["branch"]}


# ---- the same in 64 bits, plain torch ----------------------------------------------

class _Plain:
    """A branch list simulated directly: one int64 array per register, one
    complex128 amplitude per branch; an interference step sorts the children
    by key and adds equal ones."""

    def __init__(self, widths, eps, tables):
        self.dev = "cuda" if torch.cuda.is_available() else "cpu"
        self.w, self.eps = list(widths), eps
        self.reg = [torch.zeros(1, dtype=torch.int64, device=self.dev) for _ in widths]
        self.amp = torch.ones(1, dtype=torch.complex128, device=self.dev)
        self.tables = [torch.from_numpy(np.asarray(t).astype(np.int64)).to(self.dev)
                       for t in tables]

    def met(self, ctrls):
        on = torch.ones_like(self.reg[0], dtype=torch.bool)
        for c in ctrls:
            v = c[2] if len(c) > 2 else 1
            on &= ((self.reg[c[0]] >> int(c[1])) & 1) == v
        return on

    def mask(self, r):
        return (1 << self.w[r]) - 1

    def packed(self, regs):
        """Key words, unsigned order kept by flipping the top bit."""
        words = [torch.zeros_like(regs[0]), torch.zeros_like(regs[0])]
        off = 0
        for x, w in zip(regs, self.w):
            if off < 64:
                words[0] |= x << off
                if off + w > 64:
                    words[1] |= x >> (64 - off)
            else:
                words[1] |= x << (off - 64)
            off += w
        return words

    def order(self, words):
        top = -(1 << 63)
        idx = torch.sort(words[0] ^ top, stable=True)[1]
        if sum(self.w) > 64:
            idx = idx[torch.sort((words[1] ^ top)[idx], stable=True)[1]]
        return idx

    def branch(self, r, bit, u, ctrls):
        """u: four tensors or numbers u00, u01, u10, u11 per branch."""
        on = self.met(ctrls)
        bitv = 1 << int(bit)
        one = ((self.reg[r] >> int(bit)) & 1).bool()
        sel = on.nonzero().reshape(-1)
        rest = (~on).nonzero().reshape(-1)
        u = [x if isinstance(x, torch.Tensor) else torch.full_like(self.amp, x) for x in u]
        a = self.amp[sel]
        o1 = one[sel]
        c0 = torch.where(o1, u[1][sel], u[0][sel]) * a
        c1 = torch.where(o1, u[3][sel], u[2][sel]) * a
        regs = [torch.cat([x[rest], x[sel], x[sel]]) for x in self.reg]
        base = self.reg[r][sel] & ~bitv
        regs[r] = torch.cat([self.reg[r][rest], base, base | bitv])
        amp = torch.cat([self.amp[rest], c0, c1])
        words = self.packed(regs)
        idx = self.order(words)
        w0, w1 = words[0][idx], words[1][idx]
        new = torch.ones(idx.shape[0], dtype=torch.bool, device=self.dev)
        new[1:] = (w0[1:] != w0[:-1]) | (w1[1:] != w1[:-1])
        first = new.nonzero().reshape(-1)
        amp = amp[idx]
        out = amp[first].clone()
        nxt = first + 1
        ok = nxt < idx.shape[0]
        dup = torch.zeros_like(ok)
        dup[ok] = ~new[nxt[ok]]
        out[dup] += amp[nxt[dup]]
        keep = out.abs() >= self.eps
        self.reg = [x[idx][first][keep] for x in regs]
        self.amp = out[keep]

    def apply(self, g):
        op = g[0]
        if op == "h":
            s = math.sqrt(0.5)
            self.branch(g[1], g[2], (s, s, s, -s), g[3])
        elif op == "ry":
            c, s = math.cos(g[3] / 2), math.sin(g[3] / 2)
            self.branch(g[1], g[2], (c, -s, s, c), g[4])
        elif op == "ry_reg":
            half = (g[4] * self.reg[g[3]].double() + g[5]) * 0.5
            c, s = (torch.cos(half).to(torch.complex128), torch.sin(half).to(torch.complex128))
            self.branch(g[1], g[2], (c, -s, s, c), g[6])
        elif op == "u1q":
            m = np.asarray(g[3], np.complex128).reshape(2, 2)
            self.branch(g[1], g[2], [complex(x) for x in m.reshape(-1)], g[4])
        elif op == "x":
            self.reg[g[1]] = torch.where(self.met(g[3]), self.reg[g[1]] ^ (1 << int(g[2])),
                                         self.reg[g[1]])
        elif op == "phase":
            self.amp = torch.where(self.met(g[1]),
                                   self.amp * complex(math.cos(g[2]), math.sin(g[2])), self.amp)
        elif op in ("qload", "qunload"):
            first, count = g[1] if isinstance(g[1], tuple) else (g[1], 1)
            addr = torch.zeros_like(self.reg[0])
            off = 0
            for r in range(first, first + count):
                addr |= self.reg[r] << off
                off += self.w[r]
            t = self.tables[g[3]]
            inside = (addr >= 0) & (addr < t.shape[0])
            d = torch.where(inside, t[addr.clamp(0, t.shape[0] - 1)], torch.zeros_like(addr))
            self.reg[g[2]] = self.reg[g[2]] ^ (d & self.mask(g[2]))
        elif op == "swap":
            on = self.met(g[3])
            x, y = self.reg[g[1]], self.reg[g[2]]
            self.reg[g[1]], self.reg[g[2]] = torch.where(on, y, x), torch.where(on, x, y)
        else:
            on = self.met(g[4] if op != "mulc" else g[3])
            d = self.reg[g[1]]
            if op in ("add", "sub"):
                s = self.reg[g[2]] if g[2] >= 0 else int(g[3])
                new = d + s if op == "add" else d - s
            elif op == "muladd":
                new = d + self.reg[g[2]] * self.reg[g[3]]
            elif op == "mulc":
                c = int(g[2]) & ((1 << 64) - 1)
                new = d * (c - (1 << 64) if c >> 63 else c)
            elif op == "divxor":
                b = self.reg[g[3]]
                q = torch.where(b != 0, torch.div(self.reg[g[2]], b.clamp(min=1),
                                                  rounding_mode="floor"), torch.zeros_like(b))
                new = d ^ q
            else:
                raise ValueError(op)
            self.reg[g[1]] = torch.where(on, new & self.mask(g[1]), d)

    def marginal(self, r):
        p = torch.zeros(1 << self.w[r], dtype=torch.float64, device=self.dev)
        return p.index_add_(0, self.reg[r], self.weight()).cpu().numpy()

    def weight(self):
        return self.amp.real ** 2 + self.amp.imag ** 2

    def norm(self):
        return float(self.weight().sum())

    def export(self):
        words = self.packed(self.reg)
        idx = self.order(words)
        return {"lo": words[0][idx].cpu().numpy(), "hi": words[1][idx].cpu().numpy(),
                "amps": self.amp[idx].cpu().numpy()}


def exact(case, seed):
    f = case["family"]
    if f == "readout":
        widths = _widths(case)
        lo, hi, a = _loaded(case, seed)
        if case["fp32"]:
            a = a.astype(np.complex64).astype(np.complex128)
        p = np.abs(a.real) ** 2 + np.abs(a.imag) ** 2
        off = np.cumsum([0] + widths)

        def field(r):
            o, w = int(off[r]), widths[r]
            x = lo >> np.uint64(o) if o < 64 else hi >> np.uint64(o - 64)
            if o < 64 < o + w:
                x = x | (hi << np.uint64(64 - o))
            return x & np.uint64((1 << w) - 1)

        narrow = np.bincount(field(0).astype(np.int64), weights=p, minlength=1 << widths[0])
        values, inv = np.unique(field(1), return_inverse=True)
        return {"narrow": narrow, "values": values.view(np.int64),
                "probs": np.bincount(inv.reshape(-1), weights=p), "norm": float(p.sum())}
    circ = _circuit(case, seed)
    s = _Plain(circ["widths"], circ["eps"], circ["tables"])
    for g in circ["gates"]:
        s.apply(g)
    if f == "batch20":
        return {"addr": s.marginal(0), "inst": s.marginal(1), "data": s.marginal(2),
                "norm": s.norm()}
    if f in ("walk", "walk_batch"):
        out = {"top": s.marginal(circ["top"]), "bot": s.marginal(circ["bot"]), "norm": s.norm()}
        if "inst" in circ:
            out["inst"] = s.marginal(circ["inst"])
        elif case["n"] <= 8:
            e = s.export()
            out["system"] = _system(circ, (e["lo"], e["hi"], e["amps"]))
        return out
    if f == "arith":
        return {"narrow": s.marginal(3), "norm": s.norm()}
    out = s.export()
    if f == "circuit20":
        return _padded(out, case["cap"])
    if f == "random":
        if circ["widths"][0] <= 26:
            out["marginal"] = s.marginal(0)
        out["norm"] = s.norm()
    return out
