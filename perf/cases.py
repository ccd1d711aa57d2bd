"""The calls that users of this library make, as measured cases.

Each case names one public entry point (`paper_2501_15126_gb300._abi`), the
matrix it is given and the options it is given with.  The matrices are the
library's own synthetic ones (`paper_2501_15126_gb300.synth`): Erdos-Renyi
patterns with a forced diagonal, 0/1 or (0,1] values, the n=48 band with two
off-band nonzeros per row, and the mixed batch and request stream.

kind      the call
oneshot   permanent(): plan, compute and destroy, for one small matrix
noalloc   permanent_noalloc(): one matrix without any allocation
plan      Plan.compute() of a plan the program keeps (a whole walk, or the Gray
          sub-range [0, 2^span_log2) that checkpointed and sharded runs walk)
batch     batch(): matrices of uneven n, half 0/1 and half real, in one call
serving   Server.submit() / poll(): a burst of requests on a running server
"""
import numpy as np
import torch

from paper_2501_15126_gb300 import _abi, synth


def listed():
    return [
        # a single small integer permanent, everything included: latency of allocation, launch and copy
        {"name": "oneshot_n12_01", "kind": "oneshot", "pattern": "er", "n": 12, "p": 0.3, "values": "01"},
        # the same question from a program that may not allocate: one launch and one synchronisation
        {"name": "noalloc_n17_f64", "kind": "noalloc", "pattern": "er", "n": 17, "p": 0.3, "values": "f64"},
        # the n=24 0/1 matrix, exact: a walk of 2^23 steps that the launches weigh on
        {"name": "plan_n24_01", "kind": "plan", "pattern": "er", "n": 24, "p": 0.2, "values": "01"},
        # the same size in FP64
        {"name": "plan_n24_f64", "kind": "plan", "pattern": "er", "n": 24, "p": 0.2, "values": "f64"},
        # the largest and denser size of the batch workload, on its own: fills the GPU without code generation
        {"name": "plan_n28_f64", "kind": "plan", "pattern": "er", "n": 28, "p": 0.3, "values": "f64"},
        # double-double precision, the option for ill-conditioned real matrices; an odd size
        {"name": "plan_n23_dd", "kind": "plan", "pattern": "er", "n": 23, "p": 0.25, "values": "f64", "precision": 2},
        # the n=36 real matrix: the walk that gets its own generated kernel, whole
        {"name": "er36_f64", "kind": "plan", "pattern": "er", "n": 36, "p": 0.15, "values": "f64"},
        # a whole exact walk of a generated kernel
        {"name": "er34_01", "kind": "plan", "pattern": "er", "n": 34, "p": 0.2, "values": "01"},
        # one slice of the n=48 band run (the unit of checkpointed and sharded runs), exact
        {"name": "band48_01_slice", "kind": "plan", "pattern": "band", "n": 48, "w": 3, "extra": 2, "values": "01", "span_log2": 30},
        # the same slice in FP64
        {"name": "band48_f64_slice", "kind": "plan", "pattern": "band", "n": 48, "w": 3, "extra": 2, "values": "f64", "span_log2": 30},
        # many matrices of uneven size in one call
        {"name": "batch_mixed", "kind": "batch", "count": 500, "n_lo": 12, "n_hi": 28, "p_lo": 0.2, "p_hi": 0.4},
        # a burst of requests to a running server, most of them small
        {"name": "serving_burst", "kind": "serving", "count": 1000, "n_max": 27, "p_lo": 0.1, "p_hi": 0.3},
    ]


def draw(rng):
    kind = rng.choice(["oneshot", "noalloc", "generic", "generic", "dd", "er", "er", "band", "batch", "serving"])
    values = rng.choice(["01", "f64"])
    p = round(rng.uniform(0.12, 0.4), 3)
    if kind == "oneshot":
        return {"kind": "oneshot", "pattern": "er", "n": rng.randint(6, 18), "p": p, "values": values}
    if kind == "noalloc":
        return {"kind": "noalloc", "pattern": "er", "n": rng.randint(9, 27), "p": p, "values": values}
    if kind == "generic":
        return {"kind": "plan", "pattern": "er", "n": rng.randint(13, 30), "p": p, "values": values}
    if kind == "dd":
        return {"kind": "plan", "pattern": "er", "n": rng.randint(15, 25), "p": p, "values": "f64", "precision": 2}
    if kind == "er":
        return {"kind": "plan", "pattern": "er", "n": rng.randint(31, 35), "p": round(rng.uniform(0.1, 0.2), 3), "values": values}
    if kind == "band":
        return {"kind": "plan", "pattern": "band", "n": rng.randint(37, 48), "w": rng.randint(2, 3), "extra": rng.randint(1, 2),
                "values": values, "span_log2": rng.randint(24, 30)}
    if kind == "batch":
        lo = rng.randint(9, 20)
        return {"kind": "batch", "count": int(2 ** rng.uniform(4, 9)), "n_lo": lo, "n_hi": rng.randint(lo, 28),
                "p_lo": 0.2, "p_hi": 0.4}
    return {"kind": "serving", "count": int(2 ** rng.uniform(4, 10)), "n_max": rng.randint(20, 27), "p_lo": 0.1, "p_hi": 0.3}


def _matrices(case, seed):
    """The dense matrices of a case, from the seed alone."""
    if case["kind"] == "batch":
        return [item.a for item in synth.batch(case["count"], case["n_lo"], case["n_hi"], case["p_lo"], case["p_hi"], seed=seed)]
    if case["kind"] == "serving":
        stream = synth.serving_stream(rate=2000.0, duration=2.0, seed=seed, p_lo=case["p_lo"], p_hi=case["p_hi"],
                                      n_max=case["n_max"], limit=case["count"])
        return [request.a for request in stream]
    if case["pattern"] == "band":
        return [synth.band_plus(case["n"], case["w"], case["extra"], seed=seed, values=case["values"])]
    return [synth.single_er(case["n"], case["p"], seed, values=case["values"], shuffle_cols=True)]


def prepare(case, seed):
    state = {"kind": case["kind"], "precision": case.get("precision", 0),
             "matrices": [_abi.CSRMatrix(a) for a in _matrices(case, seed)]}
    if case["kind"] == "plan":
        options = {"precision": state["precision"]}
        if "span_log2" in case:
            options["g_hi"] = 1 << case["span_log2"]
        state["slice"] = "span_log2" in case
        state["plan"] = _abi.Plan(state["matrices"][0], **options)
    if case["kind"] == "serving":
        state["server"] = _abi.Server()
    return state


def run(state):
    kind, stream = state["kind"], torch.cuda.current_stream().cuda_stream
    if kind == "plan":
        results = [state["plan"].compute(stream)]
    elif kind == "oneshot":
        results = [_abi.permanent(state["matrices"][0], stream)]
    elif kind == "noalloc":
        results = [_abi.permanent_noalloc(state["matrices"][0], stream)]
    elif kind == "batch":
        results = _abi.batch(state["matrices"], stream=stream)
    else:
        server = state["server"]
        tickets = [server.submit(m) for m in state["matrices"]]
        results = [server.poll(t) for t in tickets]
    return _outputs(results, state.get("slice", False), state["precision"] == 2)


def _outputs(results, is_slice, is_dd):
    """What the calls computed: statuses; exact integers as 64-bit words; FP64 permanents (the rounded sum of
    the pair, and what the rounding left of it where double-double was asked for) and their sums of |terms|,
    which the library accumulates in FP32."""
    out = {"status": np.array([r.status for r in results], dtype=np.int64)}
    if any(r.vtype == _abi.PERM_I64 for r in results):   # (zeros in the places of real matrices)
        words = [list(r.partial) if is_slice else [r.i128_lo, r.i128_hi & ((1 << 64) - 1)] for r in results]
        out["words"] = np.array(words, dtype=np.uint64).view(np.int64)
    if any(r.vtype == _abi.PERM_F64 for r in results):   # (zeros in the places of integer matrices)
        hi, lo = np.array([r.f64 for r in results]), np.array([r.f64_lo for r in results])
        out["value"] = hi + lo
        if is_dd:
            out["value_lo"] = (hi - out["value"]) + lo
        out["abs_terms"] = np.array([r.abs_term_sum for r in results], dtype=np.float32)
    return out


def work(case):
    """Bytes: the matrices and the results once.  Operations: one per term of the signed sum over the
    2^(n-1) Gray indices (products shared between terms are not counted)."""
    ms = _matrices(case, 1)
    nnz = sum(int(np.count_nonzero(a)) for a in ms)
    rows = sum(a.shape[0] for a in ms)
    steps = sum(2.0 ** (case["span_log2"] if "span_log2" in case else a.shape[0] - 1) for a in ms)
    return {"bytes": 12.0 * nnz + 4.0 * (rows + len(ms)) + 32.0 * len(ms), "flops": steps}


def _row_expansion(a, device):
    """perm(a), a >= 0, row by row over the sets of columns taken (Eq. 1): every term is positive, so the FP64
    sum is good to a few units in the last place.  None where the sets would not fit."""
    n = a.shape[0]
    if n > (28 if device == "cuda" else 20):
        return None
    f = torch.zeros(1 << n, dtype=torch.float64, device=device)
    f[0] = 1.0
    for i in range(n):
        g = torch.zeros_like(f)
        for j in np.flatnonzero(a[i]):
            fv, gv = f.view(-1, 2, 1 << int(j)), g.view(-1, 2, 1 << int(j))
            gv[:, 1].add_(fv[:, 0], alpha=float(a[i, j]))
        f = g
    return float(f[-1])


def _frontier_expansion(a, device, most=1 << 26):
    """The same expansion for sparse matrices of any n, over the sets of taken columns that a later row can still
    take (equal sets merged).  None beyond `most` sets."""
    n = a.shape[0]
    nz, left, order, seen = a != 0, list(range(a.shape[0])), [], np.zeros(a.shape[0], dtype=bool)
    while left:   # next the row that opens the fewest new columns, ties by those it closes
        def growth(i):
            later = nz[[r for r in left if r != i]].any(axis=0) if len(left) > 1 else np.zeros(n, dtype=bool)
            return int((later & (seen | nz[i])).sum())
        i = min(left, key=growth)
        left.remove(i)
        order.append(i)
        seen |= nz[i]
    sets = torch.zeros(1, dtype=torch.int64, device=device)
    vals = torch.ones(1, dtype=torch.float64, device=device)
    for k, i in enumerate(order):
        later = nz[order[k + 1:]].any(axis=0) if k + 1 < n else np.zeros(n, dtype=bool)
        keep = sum(1 << j for j in range(n) if later[j])
        must = sum(1 << j for j in range(n) if not later[j] and nz[order[:k + 1], j].any()
                   and nz[order[k:], j].any())   # columns that close with this row have to be taken by now
        new_sets, new_vals = [], []
        for j in np.flatnonzero(nz[i]):
            bit = 1 << int(j)
            free = (sets & bit) == 0
            s = sets[free] | bit
            v = vals[free] * float(a[i, j])
            ok = (s & must) == must
            new_sets.append(s[ok] & keep)
            new_vals.append(v[ok])
        s, v = torch.cat(new_sets), torch.cat(new_vals)
        if s.numel() == 0:
            return 0.0
        if s.numel() > most:
            return None
        sets, inverse = torch.unique(s, return_inverse=True)
        vals = torch.zeros(sets.numel(), dtype=torch.float64, device=device).index_add_(0, inverse, v)
    return float(vals.sum())


def exact(case, seed):
    if "span_log2" in case:
        return None   # a slice's partial sum belongs to the column order the library picks
    device = "cuda" if torch.cuda.is_available() else "cpu"
    matrices = _matrices(case, seed)
    if all(a.dtype != np.float64 for a in matrices):
        return None   # integers are compared as they are
    got = []
    for a in matrices:
        v = 0.0   # an integer matrix has no FP64 value
        if a.dtype == np.float64:
            v = _row_expansion(a, device)
            if v is None:
                v = _frontier_expansion(a, device, 1 << 26 if device == "cuda" else 1 << 20)
        if v is None:
            return None
        got.append(v)
    out = {"value": np.array(got), "status": None, "abs_terms": None}
    if any(a.dtype != np.float64 for a in matrices):
        out["words"] = None
    if case.get("precision", 0) == 2:
        out["value_lo"] = None
    return out
