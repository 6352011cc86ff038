"""Timed cases of the library: the calls that its users make, over their real range.

Two kinds.  "amplitudes": one Plan.contract_amplitudes call, the hot path (slice
selection, the chain of pairwise contractions, the cross-slice FP64 sum), from the
smallest circuit of the smoke test to a slice range of the largest configured one.
"pair": one contract_pair call with the library's own choice of kernel, the
building block of that chain, at the sizes and index orders of the pairwise
benchmark and tests.  All extents are powers of two (every index has dimension 2),
so a case gives log2 of M, N and K; ragged are the splits between them and the
index orders.
"""
import weakref

import numpy as np
import torch

import paper_2110_14502_gb300 as T

_MASK = (1 << 64) - 1


def _amp(name, rows, cols, depth, cseed, num_open, num_sliced, width_cap, nb, slices, precision, io):
    return dict(name=name, kind="amplitudes", rows=rows, cols=cols, depth=depth, cseed=cseed, num_open=num_open,
                num_sliced=num_sliced, width_cap=width_cap, nb=nb, slices=slices, precision=precision, io=io)


def _pair(name, nm, nn, nk, order, precision, oseed=1):
    return dict(name=name, kind="pair", nm=nm, nn=nn, nk=nk, order=order, oseed=oseed, precision=precision)


def listed():
    return [
        # the smoke test's circuit, one small request: 37 tiny steps, where launches and host time count
        _amp("amp_4x4_c64", 4, 4, 8, 1, 6, -1, 0, 1, -1, "c64", "host"),
        # a typical serving request (5x5, 256 amplitudes for each of two bitstrings), replayed as the server does
        _amp("amp_5x5_split_bf16_graph", 5, 5, 12, 7, 8, -1, 0, 2, -1, "split_bf16", "graph"),
        # the 30-qubit sub-case of the 6x6 configuration: every one of its 1024 slices, 4 batches of 64 amplitudes
        _amp("amp_5x6_scaled_fp16", 5, 6, 16, 2, 6, 10, 0, 4, -1, "scaled_fp16", "host"),
        # the benchmark's 8x8 configuration in its default precision, a leading range of its slices
        _amp("amp_8x8_split_fp16", 8, 8, 20, 4, 10, -1, 26, 1, 128, "split_fp16", "device"),
        # the smallest tensor-core step (the smoke test's): operand split, GEMM and the error check per call
        _pair("pair_8_7_6_split_bf16", 8, 7, 6, "random", "split_bf16"),
        # an ordinary dense step with unordered indices, as the pairwise benchmark draws them
        _pair("pair_12_12_10_split_fp16", 12, 12, 10, "random", "split_fp16"),
        # the dense compute-bound step in the planner's layout
        _pair("pair_13_13_12_split_bf16", 13, 13, 12, "planner", "split_bf16"),
        # a wide tensor against a narrow one over a long contracted index: the operand dominates (4 GiB)
        _pair("pair_16_6_13_split_fp16", 16, 6, 13, "random", "split_fp16"),
        # a short contracted index: the output dominates (2 GiB), 16-bit scaled products
        _pair("pair_14_14_5_scaled_bf16", 14, 14, 5, "random", "scaled_bf16"),
        # the plain complex64 GEMM on the FP32 cores in the planner's layout
        _pair("pair_12_12_9_c64", 12, 12, 9, "planner", "c64"),
        # a vector-like step: a high-rank tensor streamed against a rank-7 one, unordered indices
        _pair("pair_22_3_4_c64", 22, 3, 4, "random", "c64"),
        # the last step of a slice: two wide tensors contracted into a small open batch
        _pair("pair_3_3_18_c64", 3, 3, 18, "planner", "c64"),
    ]


def draw(rng):
    precisions = ["c64", "split_bf16", "split_fp16", "scaled_fp16", "scaled_bf16"]
    if rng.random() < 0.35:
        rows = rng.randint(3, 5)
        cols = max(3, min(5, rows + rng.randint(-1, 1)))
        depth = rng.randint(6, 14)
        return dict(kind="amplitudes", rows=rows, cols=cols, depth=depth, cseed=rng.randint(1, 1 << 30),
                    num_open=rng.randint(0, min(9, rows * cols - 1)), num_sliced=rng.choice([-1, 1, 2, 3, 5]),
                    width_cap=0, nb=int(2 ** rng.uniform(0, 3.99)), slices=-1, precision=rng.choice(precisions),
                    io=rng.choice(["host", "device", "graph"]))
    what = rng.choice(["dense", "dense", "wide_a", "expand", "stream", "dot"])
    precision = rng.choice(precisions)
    if what == "dense":
        nm, nn = rng.randint(7, 13), rng.randint(4, 13)
        nk = rng.randint(3, 12)
        nk = max(3, min(nk, (32 if precision == "c64" else 36) - nm - nn))
    elif what == "wide_a":
        nm, nn = rng.randint(13, 17), rng.randint(4, 7)
        nk = rng.randint(3, 27 - nm)
    elif what == "expand":
        nm, nn, nk = rng.randint(9, 14), rng.randint(7, 13), rng.randint(0, 5)
    elif what == "stream":
        nm, nn, nk = rng.randint(8, 22), rng.randint(0, 4), rng.randint(0, 4)
    else:
        nm = rng.randint(0, 6)
        nn, nk = rng.randint(0, 6 - nm), rng.randint(8, 19)
    return dict(kind="pair", nm=nm, nn=nn, nk=nk, order=rng.choice(["random", "planner"]),
                oseed=rng.randint(1, 1 << 30), precision=precision)


# ---- amplitudes --------------------------------------------------------------

# A program keeps a circuit's plan and passes it new bitstrings: the states of one
# case share the plan while any of them is alive.
_plans = weakref.WeakValueDictionary()


def _plan(case):
    key = tuple(case[k] for k in ("rows", "cols", "depth", "cseed", "num_open", "num_sliced", "width_cap"))
    p = _plans.get(key)
    if p is None:
        n = case["rows"] * case["cols"]
        c = T.random_circuit(case["rows"], case["cols"], case["depth"], case["cseed"])
        net = T.build_network(c, list(range(n - case["num_open"], n)))
        p = T.plan(net, num_sliced=case["num_sliced"], max_log2_intermediate=case["width_cap"], search_trials=16, seed=1)
        _plans[key] = p
    return p


def _bitstrings(case, seed):
    n = case["rows"] * case["cols"]
    w = np.random.default_rng([seed, 11]).integers(0, 1 << 64, size=(case["nb"], 1), dtype=np.uint64)
    return w & np.uint64((1 << n) - 1)


# ---- pairs -------------------------------------------------------------------

def _labels(case):
    """Index labels of A, B, C, slowest first: "planner" keeps the contracted ones innermost in one order, as the
    planner lays its tensors out; "random" draws all three orders."""
    nm, nn, nk = case["nm"], case["nn"], case["nk"]
    x = list(range(nm + nn + nk))
    m, n, k = x[:nm], x[nm:nm + nn], x[nm + nn:]
    if case["order"] == "planner":
        return m + k, n + k, m + n
    rng = np.random.default_rng([case["oseed"], nm, nn, nk])
    return tuple([int(v) for v in rng.permutation(s)] for s in (m + k, n + k, m + n))


def _randn(count, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    return torch.randn(count, dtype=torch.complex64, device="cuda", generator=g)


def prepare(case, seed):
    if case["kind"] == "pair":
        la, lb, lc = _labels(case)
        return dict(kind="pair", A=_randn(1 << len(la), 2 * seed + 1), B=_randn(1 << len(lb), 2 * seed + 2),
                    C=torch.empty(1 << len(lc), dtype=torch.complex64, device="cuda"), la=la, lb=lb, lc=lc,
                    precision=case["precision"])
    words = _bitstrings(case, seed)
    state = dict(kind="amplitudes", plan=_plan(case), precision=case["precision"], slices=case["slices"],
                 io=case["io"], words=words)
    if case["io"] != "host":
        state["words"] = torch.from_numpy(words.view(np.int64)).cuda()
        state["out"] = torch.empty((case["nb"] << case["num_open"]) * 2, dtype=torch.float64, device="cuda")
        state["stream"] = torch.cuda.Stream()
    return state


def run(state):
    s = state
    if s["kind"] == "pair":
        return T.contract_pair(s["A"], s["la"], s["B"], s["lb"], s["C"], s["lc"], precision=s["precision"])
    if s["io"] == "host":
        return s["plan"].contract_amplitudes(s["words"], precision=s["precision"], slice_count=s["slices"])
    return s["plan"].contract_amplitudes(s["words"], precision=s["precision"], slice_count=s["slices"], out=s["out"],
                                         stream=s["stream"], use_graph=1 if s["io"] == "graph" else 0)


def work(case):
    if case["kind"] == "pair":
        m, n, k = 1 << case["nm"], 1 << case["nn"], 1 << case["nk"]
        return {"bytes": 8 * (m * k + k * n + m * n), "flops": 8 * m * n * k}
    info = _plan(case).info()
    slices = info["num_slices"] if case["slices"] < 0 else case["slices"]
    # one bitstring's contraction of every slice: what several bitstrings can share differs between plans
    return {"bytes": 8 * case["nb"] + 16 * (case["nb"] << case["num_open"]), "flops": info["flops_per_slice"] * slices}


# ---- the same results in 64 bits, without the library ------------------------

def _offsets(labels, group):
    """Element offset, in a tensor with these labels, of every value of the group's bits (its last label fastest)."""
    o = torch.zeros(1, dtype=torch.int64, device="cuda")
    for l in group:
        st = 1 << (len(labels) - 1 - labels.index(l))
        o = (o[:, None] + torch.tensor([0, st], device="cuda")[None, :]).reshape(-1)
    return o


def _exact_pair(case, seed):
    s = prepare(case, seed)
    la, lb, lc = s["la"], s["lb"], s["lc"]
    m = [l for l in la if l in lc]
    k = [l for l in la if l not in lc]
    n = [l for l in lb if l in lc]
    am, ak, bk, bn, cm, cn = (_offsets(*x) for x in ((la, m), (la, k), (lb, k), (lb, n), (lc, m), (lc, n)))
    B = s["B"][(bk[:, None] + bn[None, :])].to(torch.complex128)
    C = torch.empty(1 << len(lc), dtype=torch.complex128, device="cuda")
    step = max(1, (1 << 26) // max(ak.numel(), bn.numel()))
    for i in range(0, am.numel(), step):
        A = s["A"][am[i:i + step, None] + ak[None, :]].to(torch.complex128)
        C[cm[i:i + step, None] + cn[None, :]] = A @ B
    return C


def _gates(rows, cols, depth, seed):
    """The circuit protocol: a layer of one-qubit gates, then `depth` cycles of an fSim(pi/2, pi/6) layer on coupler
    pattern A, B, C, D (horizontal even, odd, vertical even, odd) and a one-qubit layer; SplitMix64 draws."""
    state = seed & _MASK

    def uniform(k):
        nonlocal state
        state = (state + 0x9E3779B97F4A7C15) & _MASK
        z = state
        z = ((z ^ (z >> 30)) * 0xBF58476D1CE4E5B9) & _MASK
        z = ((z ^ (z >> 27)) * 0x94D049BB133111EB) & _MASK
        return (((z ^ (z >> 31)) >> 32) * k) >> 32

    w = np.exp(1j * np.pi / 4)
    one = [np.array(u) / np.sqrt(2) for u in ([[1, -1j], [-1j, 1]], [[1, -1], [1, 1]], [[1, -w], [1 / w, 1]])]
    fsim = np.diag([1, 0, 0, np.exp(-1j * np.pi / 6)]).astype(complex)
    fsim[1, 2] = fsim[2, 1] = -1j
    n, prev, out = rows * cols, {}, []

    def layer():
        for q in range(n):
            kinds = [x for x in range(3) if x != prev.get(q)]
            prev[q] = kinds[uniform(len(kinds))]
            out.append(((q,), one[prev[q]]))

    layer()
    for c in range(depth):
        p = c % 4
        if p < 2:
            pairs = [(r * cols + x, r * cols + x + 1) for r in range(rows) for x in range(p, cols - 1, 2)]
        else:
            pairs = [(r * cols + x, (r + 1) * cols + x) for r in range(p - 2, rows - 1, 2) for x in range(cols)]
        out += [(ab, fsim) for ab in pairs]
        layer()
    return out


def _exact_amplitudes(case, seed):
    n, k = case["rows"] * case["cols"], case["num_open"]
    if n > 30 or case["slices"] >= 0:
        return None  # no state vector of that size, and a leading range of slices is no amplitude
    psi = torch.zeros(1 << n, dtype=torch.complex128, device="cuda")
    psi[0] = 1.0
    pending = [np.eye(2, dtype=complex) for _ in range(n)]  # one-qubit gates wait for their qubit's next pair

    def apply(a, b, u):
        nonlocal psi
        v = psi.view(1 << (n - 1 - b), 2, 1 << (b - 1 - a), 2, 1 << a)  # axes: high, x_b, middle, x_a, low
        x = v.permute(3, 1, 0, 2, 4).reshape(4, -1)
        x = torch.from_numpy(np.ascontiguousarray(u)).cuda() @ x
        psi = x.view(2, 2, v.shape[0], v.shape[2], v.shape[4]).permute(2, 1, 3, 0, 4).reshape(-1)

    for qs, u in _gates(case["rows"], case["cols"], case["depth"], case["cseed"]):
        if len(qs) == 1:
            pending[qs[0]] = u @ pending[qs[0]]
        else:
            a, b = qs
            apply(a, b, u @ np.kron(pending[a], pending[b]))
            pending[a] = pending[b] = np.eye(2, dtype=complex)
    for a in range(0, n - 1, 2):
        apply(a, a + 1, np.kron(pending[a], pending[a + 1]))
    if n % 2:
        apply(n - 2, n - 1, np.kron(np.eye(2), pending[n - 1]))
    w = torch.from_numpy(_bitstrings(case, seed).astype(np.int64)[:, 0]).cuda() & ((1 << (n - k)) - 1)
    return psi[w[:, None] | (torch.arange(1 << k, device="cuda")[None, :] << (n - k))]


def exact(case, seed):
    return _exact_pair(case, seed) if case["kind"] == "pair" else _exact_amplitudes(case, seed)
