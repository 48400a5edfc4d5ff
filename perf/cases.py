"""The calls whose speed this repository is measured by.

Every case goes through the package's public entry points (plan, contract, xeb, spoof,
rejection_sample, slice_cut) on seeded Sycamore-style circuits, at the sizes of the tests,
the benchmark and the server's requests: 12 to 40 qubits, 8 to 16 cycles, one to 16384
batches, in the three precisions, over all slices, a few partial assignments of a cut, or
one chunk of a sampling job.

A case is a dict; its "kind" selects the call:

* contract   batches of 2^n_open amplitudes over a slice set: what tn_sample and every
             sampling job spend their time on (the sampler draws from these amplitudes)
* xeb        the amplitudes of given bitstrings and their linear XEB (verification)
* spoof      one batch's N most probable strings (XEB spoofing)
* sampler    the accept / pick step on a job's batch probabilities
* slice_cut  the cut of the sorted slice norms (selection)
"""
import functools
import math

import numpy as np
import torch

import paper_2112_15083_gb300 as tn
from paper_2112_15083_gb300 import circuits

PREC = {"c64": tn.tn.PREC_C64, "bf16x2": tn.tn.PREC_BF16X2, "fp16x2": tn.tn.PREC_FP16X2}

# Order-search trials by grid (rows, cols): the larger networks are searched longer, as
# the benchmark does.
TRIALS = {(4, 7): 128, (5, 8): 256}


def listed():
    return [
        # the smallest call: a 12-qubit circuit's 16 batches, bound by launches
        dict(name="amps_12q_c64", kind="contract", rows=3, cols=4, cycles=8, sliced=2, open=6, prec="c64",
             log2_batches=4, batches=16, slices="all", host=False),
        # a served request in several small groups with a ragged last one, at partial
        # fidelity (three assignments of a four-leg cut), on host arrays
        dict(name="amps_20q_c64_ragged", kind="contract", rows=4, cols=5, cycles=10, sliced=8, open=6, prec="c64",
             log2_batches=8, batches=1000, slices="cut3", host=True),
        # one group of a mid-sized request in each tensor-core format
        dict(name="amps_20q_bf16", kind="contract", rows=4, cols=5, cycles=12, sliced=6, open=6, prec="bf16x2",
             log2_batches=10, batches=1024, slices="all", host=False),
        dict(name="amps_24q_fp16", kind="contract", rows=4, cols=6, cycles=12, sliced=8, open=6, prec="fp16x2",
             log2_batches=12, batches=4000, slices="all", host=False),
        # verification of 1000 samples of a 24-qubit circuit
        dict(name="xeb_24q_c64", kind="xeb", rows=4, cols=6, cycles=12, sliced=8, open=6, prec="c64",
             log2_batches=10, strings=1000),
        # spoofing: a tenth of one batch of 2^16 strings
        dict(name="spoof_20q_c64", kind="spoof", rows=4, cols=5, cycles=12, sliced=6, open=16, prec="c64",
             log2_batches=0, strings=6553),
        # the 28-qubit workload at fidelity 1: one job of five groups of 16384 batches in
        # split bf16, one group in complex64 (the library's default precision)
        dict(name="amps_28q_bf16", kind="contract", rows=4, cols=7, cycles=14, sliced=10, open=6, prec="bf16x2",
             log2_batches=14, batches=81920, slices="all", host=False),
        dict(name="amps_28q_c64", kind="contract", rows=4, cols=7, cycles=14, sliced=10, open=6, prec="c64",
             log2_batches=14, batches=16384, slices="all", host=False),
        # a chunk of the 40-qubit sampling job: eight slices, a part of its batch groups
        dict(name="chunk_40q_bf16", kind="contract", rows=5, cols=8, cycles=16, cap=30, open=6, prec="bf16x2",
             log2_batches=12, batches=81920, slices="chunk3", host=False, groups=55),
        # the final pass of that job: accept / pick over all of its batches
        dict(name="sampler_40q", kind="sampler", b_bits=34, batches=225280, alpha=2.0),
        # the cut at f = 1/64 (2^9 norms), and at the largest size the call takes
        dict(name="slice_cut_9", kind="slice_cut", k=9, f=1.0 / 64),
        dict(name="slice_cut_12", kind="slice_cut", k=12, f=0.3),
    ]


def draw(rng):
    kind = rng.choices(["contract", "chunk", "xeb", "spoof", "sampler", "slice_cut"], [10, 2, 2, 1, 1, 1])[0]
    if kind == "sampler":
        return dict(kind="sampler", b_bits=rng.randint(6, 50), batches=int(math.exp(rng.uniform(0.0, math.log(225280)))),
                    alpha=rng.choice([1.5, 2.0, 4.0]))
    if kind == "slice_cut":
        return dict(kind="slice_cut", k=rng.randint(3, 12), f=rng.choice([0.01, 0.05, 0.3, 0.9]))
    if kind == "chunk":
        groups = rng.randint(1, 19)
        return dict(kind="contract", rows=5, cols=8, cycles=16, cap=30, open=6, prec=rng.choice(["bf16x2", "fp16x2"]),
                    log2_batches=12, batches=4096 * groups + rng.randint(1, 4096),
                    slices=rng.choice(["chunk0", "chunk1", "chunk2", "chunk3"]), host=False, groups=55, circuit_seed=rng.randint(1, 999))
    rows, cols, sliced = rng.choice([(3, 4, 2), (4, 4, 4), (4, 5, 6), (4, 6, 8), (4, 7, 10)])
    cycles = 14 if rows * cols == 28 else rng.randint(8, 12)
    prec = rng.choice(["c64", "bf16x2", "fp16x2"])
    case = dict(kind=kind, rows=rows, cols=cols, cycles=cycles, sliced=sliced, open=6, prec=prec,
                circuit_seed=rng.randint(0, 999))
    if kind == "spoof":
        n_open = rng.randint(8, min(16, rows * cols - 2))
        return dict(case, open=n_open, prec="c64", log2_batches=0, strings=max(1, int((1 << n_open) * 0.1)))
    n = int(math.exp(rng.uniform(math.log(3.0), math.log(20000.0))))
    # the server's rule: the smallest group of at least the request's batches, 2^8 to 2^14
    lb = max(8, min(14, math.ceil(math.log2(n))))
    if rows * cols == 28:
        lb = 14
    if kind == "xeb":
        return dict(case, prec="c64" if rows * cols < 28 else "bf16x2", log2_batches=min(lb, 10 if rows * cols < 28 else 14),
                    strings=min(n, 4000))
    return dict(case, log2_batches=lb, batches=n, slices=rng.choice(["all", "all", "cut3"]) if rows * cols < 28 else "all",
                host=rng.random() < 0.3)


# ------------------------------------------------------------------ inputs


def _circuit(case):
    return circuits.sycamore_grid(case["rows"], case["cols"], case["cycles"], seed=case.get("circuit_seed", 0))


def _open(case):
    return circuits.default_open_qubits(case["rows"], case["cols"], case["open"])


def _cut_legs(case):
    """The sliced legs of the partial-fidelity cases: a four-leg cut (the first qubits' wires
    in the middle of the circuit), then further legs that every slice set is closed under."""
    n = case["rows"] * case["cols"]
    count = [0] * n
    for g in _circuit(case).gates:
        if len(g.qubits) == 2:
            for q in g.qubits:
                count[q] += 1
    legs = [(q, max(1, count[q] // 2)) for q in range(n) if count[q] >= 2]
    return legs[: min(max(5, case["sliced"]), len(legs))]


def _cut_patterns(seed):
    """Three of the 16 partial assignments of the cut (the dominant ones differ by input)."""
    return sorted(int(x) for x in np.random.default_rng(1000 + seed).choice(16, size=3, replace=False))


def _plan_args(case):
    kw = dict(log2_batches=case["log2_batches"], precision=PREC[case["prec"]], hbm_budget_bytes=90e9,
              order_trials=TRIALS.get((case["rows"], case["cols"]), 64))
    if "cap" in case:
        kw.update(max_log2_tensor=case["cap"], job_groups=case["groups"], anneal_iters=2000)
    elif case.get("slices") == "cut3":
        kw.update(sliced=_cut_legs(case), parallel_search=True)
    else:
        kw.update(n_auto_sliced=case["sliced"], parallel_search=True)
    return kw


def _chunk(plan, seed, log2_chunk):
    """2^log2_chunk slices that differ in the legs which add the least work when they vary
    inside the chunk, as a sampling job picks them; the other legs' values come from the seed."""
    n = len(plan.sliced_edges())
    base = int(np.random.default_rng(2000 + seed).integers(0, 1 << n))
    legs = []
    for _ in range(log2_chunk):
        cost = []
        for e in range(n):
            if e not in legs:
                cost.append((plan.estimate(_subcube(base, legs + [e]))[1], e))
        legs.append(min(cost)[1])
    return _subcube(base, legs)


def _subcube(base, legs):
    out = [base]
    for e in legs:
        out = [s & ~(1 << e) for s in out] + [s | (1 << e) for s in out]
    return np.array(sorted(out), dtype=np.uint64)


def _slices(case, plan, seed):
    if case.get("slices", "all") == "all":
        return np.arange(1 << len(plan.sliced_edges()), dtype=np.uint64)
    if case["slices"] == "cut3":
        free = len(_cut_legs(case)) - 4
        return np.array([x | (r << 4) for x in _cut_patterns(seed) for r in range(1 << free)], dtype=np.uint64)
    return _chunk(plan, seed, int(case["slices"][len("chunk"):]))


def _closed(case, seed):
    return circuits.random_closed_bits(case["batches"], case["rows"] * case["cols"] - case["open"], 3000 + seed)


def _strings(case, seed):
    return np.random.default_rng(4000 + seed).integers(0, 1 << (case["rows"] * case["cols"]), size=case["strings"],
                                                       dtype=np.uint64)


def _pattern(case, seed):
    return int(np.random.default_rng(5000 + seed).integers(0, 1 << (case["rows"] * case["cols"] - case["open"])))


def _norms(case, seed):
    # the same norms in another order for each input, so that the cut keeps as many of them
    r = np.random.default_rng(6000).exponential(size=1 << case["k"])
    return np.random.default_rng(6001 + seed).permutation(r / r.sum())


def prepare(case, seed):
    kind = case["kind"]
    if kind == "sampler":
        g = torch.Generator(device="cuda").manual_seed(7000 + seed)
        # Porter-Thomas batch probabilities
        p = torch.empty((case["batches"], 64), dtype=torch.float64, device="cuda").exponential_(generator=g)
        return dict(case=case, p=p * 2.0 ** -(case["b_bits"] + 6), seed=seed)
    if kind == "slice_cut":
        return dict(case=case, R=_norms(case, seed))
    plan = tn.plan(tn.circuit_load(_circuit(case).serialize()), _open(case), **_plan_args(case))
    st = dict(case=case, plan=plan, slices=_slices(case, plan, seed))
    if kind == "contract":
        cb = _closed(case, seed)
        st["closed"] = cb if case["host"] else torch.from_numpy(cb.astype(np.int64)).cuda()
        if not case["host"]:
            st["out"] = torch.empty((case["batches"], 1 << case["open"]), dtype=torch.complex128, device="cuda")
    elif kind == "xeb":
        st["strings"] = _strings(case, seed)
    else:
        st["pattern"] = _pattern(case, seed)
    return st


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "sampler":
        return tn.rejection_sample(state["p"], case["b_bits"], case["alpha"], state["seed"])
    if kind == "slice_cut":
        return tn.slice_cut(state["R"], case["f"])
    if kind == "contract":
        return state["plan"].contract(state["slices"], state["closed"], out=state.get("out"))
    if kind == "xeb":
        return state["plan"].xeb(state["slices"], state["strings"], return_amplitudes=True)
    return state["plan"].spoof(state["slices"], state["pattern"], case["strings"], return_probs=True)


# ------------------------------------------------------------------ work


@functools.lru_cache(maxsize=None)
def _flops(items):
    """Multiply-adds of the plan's contraction tree: the batch-independent products once (the
    slices of a chunk share most of them: the legs that vary inside it are chosen so), the
    others once per batch group and value of the sliced legs they depend on."""
    case = dict(items)
    info, steps, _ = tn.tn.plan_host(tn.circuit_load(_circuit(case).serialize()), _open(case), **_plan_args(case))
    groups = -(-case.get("batches", case.get("strings", 1)) // (1 << case["log2_batches"]))
    if case["kind"] == "spoof":
        groups = 1
    # a plan over all slices counts them in the products' sizes already
    in_sizes = info["flops_per_slice"] >= 0.999 * info["flops_all_slices"]
    n = {"all": 1 << info["n_sliced"], "cut3": 3 << max(0, info["n_sliced"] - 4)}.get(case.get("slices", "all"))
    if n is None:
        n = 1 << int(case["slices"][len("chunk"):])
    total = 0.0
    for bat, m, nn, k, vc, _, _ in steps.tolist():
        f = 8.0 * 2.0 ** (bat + m + nn + k) * (groups if bat >= case["log2_batches"] else 1)
        if in_sizes:
            total += f * min(1.0, n / 2.0 ** info["n_sliced"])
        else:
            total += f * (min(n, 2.0 ** vc) if bat >= case["log2_batches"] else 1)
    return total


def work(case):
    kind = case["kind"]
    if kind == "sampler":
        # the probabilities read, a flag and an index written; a sum and a prefix per value
        return {"bytes": case["batches"] * (64 * 8 + 1 + 4), "flops": case["batches"] * 64 * 2}
    if kind == "slice_cut":
        n = 1 << case["k"]
        return {"bytes": n * 8 + n * 4, "flops": n * case["k"]}
    key = tuple(sorted((k, v) for k, v in case.items() if k != "name"))
    na = 1 << case["open"]
    io = {"contract": lambda: case["batches"] * (8 + 16 * na), "xeb": lambda: case["strings"] * (8 + 16),
          "spoof": lambda: 16 * na + 16 * case["strings"]}[kind]()
    return {"bytes": io, "flops": _flops(key)}


# ------------------------------------------------------------------ exact values


def _gate2(state, n, qa, qb, U):
    """Apply a two-qubit matrix (index 2 bit(qa) + bit(qb)) to a state of 2^n in place."""
    hi, lo = max(qa, qb), min(qa, qb)
    v = state.view(1 << (n - 1 - hi), 2, 1 << (hi - 1 - lo), 2, 1 << lo)
    part = [v[:, a, :, b, :] if qa == hi else v[:, b, :, a, :] for a in (0, 1) for b in (0, 1)]
    new = []
    for i in range(4):
        acc = None
        for j in range(4):
            if U[i, j] != 0:
                acc = part[j] * complex(U[i, j]) if acc is None else acc.add_(part[j], alpha=complex(U[i, j]))
        new.append(torch.zeros_like(part[i]) if acc is None else acc)
    for i in range(4):
        part[i].copy_(new[i])


def _state(case, legs=(), values=()):
    """The final state with each leg's wire projected on its value: one 2^n vector in 64 bits.
    A leg (q, s) is qubit q's wire just before its (s+1)-th two-qubit gate."""
    n = case["rows"] * case["cols"]
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    psi = torch.zeros(1 << n, dtype=torch.complex128, device=dev)
    psi[0] = 1.0
    pend = [np.eye(2, dtype=np.complex128) for _ in range(n)]
    fixed = dict(zip(legs, values))
    seen = [0] * n
    swap = [0, 2, 1, 3]
    for g in _circuit(case).gates:
        if len(g.qubits) == 1:
            pend[g.qubits[0]] = g.matrix @ pend[g.qubits[0]]
            continue
        a, b = g.qubits
        pre = []
        for q in (a, b):
            x = pend[q]
            if (q, seen[q]) in fixed:
                x = np.diag([1.0 - fixed[(q, seen[q])], float(fixed[(q, seen[q])])]) @ x
            pre.append(x)
            pend[q] = np.eye(2, dtype=np.complex128)
            seen[q] += 1
        U = g.matrix @ np.kron(pre[0], pre[1])
        if a > b:
            _gate2(psi, n, a, b, U)
        else:
            _gate2(psi, n, b, a, U[np.ix_(swap, swap)])
    for q in range(n):
        v = psi.view(1 << (n - 1 - q), 2, 1 << q)
        x0, x1 = v[:, 0, :].clone(), v[:, 1, :].clone()
        m = pend[q]
        v[:, 0, :] = x0 * complex(m[0, 0]) + x1 * complex(m[0, 1])
        v[:, 1, :] = x0 * complex(m[1, 0]) + x1 * complex(m[1, 1])
    return psi


def _states_sum(case, seed):
    if case.get("slices", "all") == "all":
        return _state(case)
    legs = _cut_legs(case)[:4]
    psi = None
    for x in _cut_patterns(seed):
        one = _state(case, legs, [(x >> t) & 1 for t in range(4)])
        psi = one if psi is None else psi.add_(one)
    return psi


def _batch_index(case, closed):
    """Basis indices (batches, 2^n_open) of the batches with the given closed patterns."""
    n, openq = case["rows"] * case["cols"], _open(case)
    closedq = [q for q in range(n) if q not in openq]
    base = np.zeros(len(closed), dtype=np.uint64)
    for c, q in enumerate(closedq):
        base |= ((closed >> np.uint64(c)) & np.uint64(1)) << np.uint64(q)
    off = np.zeros(1 << len(openq), dtype=np.uint64)
    for r, q in enumerate(openq):
        off |= ((np.arange(1 << len(openq), dtype=np.uint64) >> np.uint64(r)) & np.uint64(1)) << np.uint64(q)
    return torch.from_numpy((base[:, None] | off[None, :]).astype(np.int64))


def exact(case, seed):
    kind = case["kind"]
    if kind == "sampler" or str(case.get("slices", "")).startswith("chunk"):
        return None  # whole numbers; a state vector of 2^40 amplitudes
    if kind == "slice_cut":
        r = np.sort(_norms(case, seed))[::-1]
        c = np.cumsum(r)
        return (None, float(c[min(len(r) - 1, int(np.searchsorted(c, case["f"])))]))
    psi = _states_sum(case, seed)
    if kind == "contract":
        return psi[_batch_index(case, _closed(case, seed)).to(psi.device)]
    if kind == "xeb":
        amps = psi[torch.from_numpy(_strings(case, seed).astype(np.int64)).to(psi.device)]
        n = case["rows"] * case["cols"]
        return (2.0 ** n * float(amps.abs().square().mean()) - 1.0, amps)
    p = psi[_batch_index(case, np.array([_pattern(case, seed)], dtype=np.uint64)).to(psi.device)].abs().square().reshape(-1)
    keep = torch.sort(torch.topk(p, case["strings"]).indices).values
    return (None, p[keep])
