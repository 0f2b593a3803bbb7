"""The framework's work as its users have it done, for timing: passes of the
loop expansion (one geometry, many tensor sets), the batched and the served
form, the combinatorial form, weight passing with rank-r expansions, strips of
infinite lattices, blocked grid contractions and the dense product under them.

``listed()`` gives the named cases, ``draw(rng)`` one more of the same ranges,
``prepare`` what a program holds before the call, ``run`` one call, ``work`` the
bytes and operations it cannot do without and ``exact`` its results in 64 bits
from plain torch or numpy."""
import ctypes
import functools
import itertools
import math

import numpy as np
import torch

from paper_2512_10910_gb300 import inputs as I
from paper_2512_10910_gb300 import pne

DTYPES = {"f64": pne.PNE_F64, "f32": pne.PNE_F32, "tf32": pne.PNE_TF32, "bf16": pne.PNE_BF16}
BETA_C = math.log(1 + math.sqrt(2)) / 2


def listed():
    return [
        # the smallest call: one 4x4 Ising network expanded to full order (its exact value), launch and host bound
        {"name": "pass_4x4_full_order", "kind": "pass", "net": "ising", "shape": "4x4", "D": 2, "sets": 1, "K": 24,
         "dtype": "f64", "arithmetic": 0, "cache": True},
        # the benchmark's step: 32 random networks of one geometry, the enumeration recomputed beside the sweeps
        {"name": "pass_16x16_D4_K8", "kind": "pass", "net": "random", "shape": "16x16", "D": 4, "sets": 32, "K": 8,
         "dtype": "f64", "arithmetic": 1, "cache": False},
        # the largest expansion: the cubic Ising lattice at order 10 and three temperatures, BF16 contractions
        {"name": "pass_8x8x8_K10_bf16", "kind": "pass", "net": "ising", "shape": "8x8x8", "D": 2, "sets": 3, "K": 10,
         "dtype": "bf16", "arithmetic": 1, "cache": False},
        # an ordinary call on an odd lattice with an odd bond dimension: FP64 sweeps, FP32 contractions, the
        # geometry's enumeration kept by the context as for any later call on it
        {"name": "pass_13x9_D5_f32", "kind": "pass", "net": "random", "shape": "13x9", "D": 5, "sets": 5, "K": 7,
         "dtype": "f32", "arithmetic": 0, "cache": True},
        # many uneven networks in one fused launch: partitions updated on new tensors, then the batch replayed
        {"name": "batch_256_uneven", "kind": "batch", "networks": 256, "mix": 1234, "K": 8, "dtype": "f64"},
        # a burst at the server: AKLT norm networks and random cubic lattices of mixed sizes and orders
        {"name": "serve_burst_24", "kind": "serve", "requests": 24, "mix": 7, "dtype": "f32"},
        # the combinatorial form over six multi-index partitions, very many tensor sets
        {"name": "comb_3x3_D4_x1024", "kind": "comb", "D": 4, "sets": 1024, "dtype": "f64"},
        # weight passing and the rank-2 expansion below T_c on the blocked Ising network, as rank-1 fails there
        {"name": "rank2_3x3_chi16", "kind": "rank_r", "block": 4, "sets": 8, "rank": 2, "form": 1, "dtype": "f64"},
        # the infinite lattice: a temperature sweep of strips up to 20 spins wide
        {"name": "strips_L10_x8", "kind": "strip", "net": "ising", "chi": 4, "L": 10, "sets": 8, "arithmetic": 1},
        # exact contraction of blocked random networks on the tensor cores
        {"name": "grid_5x4_chi16_tf32", "kind": "grid", "lx": 5, "ly": 4, "chi": 16, "sets": 32, "dtype": "tf32"},
        # the same in FP64, the reference of every expansion, at an odd bond dimension
        {"name": "grid_5x5_chi11_f64", "kind": "grid", "lx": 5, "ly": 5, "chi": 11, "sets": 3, "dtype": "f64"},
        # the dense product of one site absorption, alone
        {"name": "gemm_4x32768x256x256_bf16", "kind": "gemm", "batch": 4, "M": 32768, "N": 256, "K": 256,
         "dtype": "bf16"},
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["pass", "pass", "pass", "batch", "serve", "comb", "rank_r", "strip", "grid", "grid", "gemm",
                       "gemm"])
    any_dtype = rng.choice(["f64", "f32", "tf32", "bf16"])
    if kind == "pass":
        case = {"kind": kind, "dtype": any_dtype, "arithmetic": rng.randint(0, 1), "cache": rng.random() < 0.5}
        if rng.random() < 0.6:
            lx, ly = _log_int(rng, 3, 24), _log_int(rng, 3, 24)
            net = rng.choice(["random", "random", "ising"])
            D = 2 if net == "ising" else rng.randint(2, 6)
            most = max(1, min(64, int(3e6 / (lx * ly * D ** 4))))
            return {**case, "net": net, "shape": f"{lx}x{ly}", "D": D, "sets": _log_int(rng, 1, most),
                    "K": rng.randint(4, 8)}
        net = rng.choice(["random", "ising"])
        D = 2 if net == "ising" else rng.randint(2, 4)
        side = [rng.randint(3, 9 if D < 4 else 6) for _ in range(3)]
        K = rng.randint(4, (10 if max(side) <= 8 else 9) if net == "ising" else 8 if D < 4 else 6)
        return {**case, "net": net, "shape": "x".join(map(str, side)), "D": D, "sets": rng.randint(1, 4), "K": K}
    if kind == "batch":
        return {"kind": kind, "networks": _log_int(rng, 8, 256), "mix": rng.randint(1, 9999), "K": rng.choice([6, 8]),
                "dtype": any_dtype}
    if kind == "serve":
        return {"kind": kind, "requests": _log_int(rng, 2, 24), "mix": rng.randint(1, 9999), "dtype": any_dtype}
    if kind == "comb":
        D = rng.randint(2, 6)
        return {"kind": kind, "D": D, "sets": _log_int(rng, 1, max(1, min(1024, 3000000 // D ** 6))),
                "dtype": rng.choice(["f64", "f32"])}
    if kind == "rank_r":
        return {"kind": kind, "block": rng.randint(2, 4), "sets": _log_int(rng, 1, 8), "rank": rng.choice([1, 2, 2]),
                "form": rng.randint(0, 1), "dtype": rng.choice(["f64", "sitewise", "tf32"])}
    if kind == "strip":
        net, chi = rng.choice([("ising", 4), ("ising", 2), ("random", 3), ("random", 2)])
        return {"kind": kind, "net": net, "chi": chi, "L": rng.randint(2, 10), "sets": _log_int(rng, 1, 8),
                "arithmetic": rng.randint(0, 1)}
    dtype = rng.choice(["tf32", "bf16", "f64"])
    if kind == "grid":
        lx, ly = rng.randint(3, 6), rng.randint(3, 6)
        chi = rng.randint(2, 16 if lx < 6 else 12)
        most = (1.5e12 if dtype != "f64" else 6e10) / (2.0 * chi ** (lx + 3) * lx * ly)
        if most < 1:
            chi = 8
            most = (1.5e12 if dtype != "f64" else 6e10) / (2.0 * chi ** (lx + 3) * lx * ly)
        return {"kind": kind, "lx": lx, "ly": ly, "chi": chi, "sets": _log_int(rng, 1, max(1, min(32, int(most)))),
                "dtype": dtype}
    N, K = _log_int(rng, 16, 2048), _log_int(rng, 16, 2048)
    most = (6e11 if dtype != "f64" else 2e10) / (2.0 * N * K)
    M = _log_int(rng, 64, int(min(65536, max(64, most))))
    return {"kind": kind, "batch": _log_int(rng, 1, int(max(1, min(16, most / M)))), "M": M, "N": N, "K": K,
            "dtype": dtype}


# ---------------------------------------------------------------- inputs
class Held:
    """Values of one prepared case; library handles are released with it, last made first."""

    def __init__(self, case):
        self.case, self._release = case, []

    def own(self, destroy, handle):
        self._release.append((destroy, handle))
        return handle

    def __del__(self):
        torch.cuda.synchronize()
        while self._release:
            destroy, handle = self._release.pop()
            destroy(handle)


@functools.lru_cache(maxsize=None)
def _context():
    """The one context a program keeps for its device."""
    return pne.Context(torch.cuda.current_device())


@functools.lru_cache(maxsize=None)
def _lattice(shape, D):
    return I.square_lattice(*shape, D) if len(shape) == 2 else I.cubic_lattice(*shape, D)


def _shape(case):
    return tuple(int(x) for x in case["shape"].split("x"))


def _site_sizes(net):
    return [int(np.prod(net.leg_dims(v))) for v in range(net.n_sites)]


def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _random_flat(total, sets, seed, cubic=False):
    """Random tensor sets: U[0,1) + 0.1, or N(1, 0.3^2) on cubic lattices."""
    g = _gen(seed)
    if cubic:
        return 1.0 + 0.3 * torch.randn(sets, total, generator=g, device="cuda", dtype=torch.float64)
    return torch.rand(sets, total, generator=g, device="cuda", dtype=torch.float64) + 0.1


def _ising_flat(net, betas):
    """Square roots of the Boltzmann weights joined at each spin, one set per temperature."""
    sets = []
    for b in betas:
        p, m = math.sqrt(2 * math.cosh(b)), math.sqrt(2 * math.sinh(b))
        w = np.array([[(p + m) / 2, (p - m) / 2], [(p - m) / 2, (p + m) / 2]])
        by_degree = {}
        for k in set(np.diff(net.site_ptr).tolist()):
            by_degree[k] = sum(functools.reduce(np.multiply.outer, [w[s]] * k).reshape(-1) for s in (0, 1))
        sets.append(np.concatenate([by_degree[int(k)] for k in np.diff(net.site_ptr)]))
    return torch.from_numpy(np.stack(sets)).cuda()


def _betas(case, seed, n):
    lo, hi = (0.20, 0.25) if case.get("shape", "").count("x") == 2 else (0.30, 0.50)
    return np.random.RandomState(seed % (1 << 31)).uniform(lo, hi, n)


def _pass_data(case, seed):
    net = _lattice(_shape(case), case["D"])
    if case["net"] == "ising":
        return net, _ising_flat(net, _betas(case, seed, case["sets"]))
    return net, _random_flat(sum(_site_sizes(net)), case["sets"], seed, cubic=len(_shape(case)) == 3)


def _batch_groups(case):
    """(L, D, kinds of its networks) of every geometry of the uneven mix."""
    r = np.random.RandomState(case["mix"])
    groups = {}
    for _ in range(case["networks"]):
        L, D, ising = r.randint(6, 25), r.randint(2, 7), r.rand() < 0.5
        groups.setdefault((L, 2 if ising else D), []).append(ising)
    return sorted(groups.items())


def _batch_data(case, seed):
    out = []
    for i, ((L, D), kinds) in enumerate(_batch_groups(case)):
        net = _lattice((L, L), D)
        flat = _random_flat(sum(_site_sizes(net)), len(kinds), seed * 1009 + i)
        if any(kinds):
            betas = _betas(case, seed * 1009 + i, len(kinds))
            flat = torch.where(torch.tensor(kinds, device="cuda")[:, None], _ising_flat(net, betas), flat)
        out.append((net, (L, L), D, flat))
    return out


@functools.lru_cache(maxsize=None)
def _aklt(L):
    return I.aklt_tensors(_lattice((L, L), 4)).flat_data()[0]


def _serve_data(case, seed):
    """(network, shape, D, K, host tensors) per request: half AKLT norms L x L, half random cubic lattices."""
    r = np.random.RandomState(case["mix"])
    out = []
    for i in range(case["requests"]):
        K, L, D = int(r.randint(4, 9)), int(r.randint(8, 33)), int(r.randint(2, 5))
        if r.rand() < 0.5 and i:
            out.append((_lattice((L, L), 4), (L, L), 4, K, _aklt(L)))
        else:
            L = 6 + (L - 8) * 7 // 25
            net = _lattice((L, L, L), D)
            n = sum(_site_sizes(net))
            out.append((net, (L, L, L), D, K, np.random.default_rng([seed, i]).normal(1.0, 0.3, n)))
    return out


def _rank_r_data(case, seed):
    fractions = np.random.RandomState(seed % (1 << 31)).uniform(0.65, 0.8, case["sets"])
    nets = [I.ising_blocked(3, 3, case["block"], BETA_C / f) for f in fractions]
    parts = I.square3x3_six_lines() if case["form"] else I.square3x3_pinwheel()
    return nets, parts


def _strip_data(case, seed):
    r = np.random.RandomState(seed % (1 << 31))
    chi, n = case["chi"], case["sets"]
    if case["net"] == "ising":
        betas = r.uniform(0.25, 0.42, n)
        return torch.from_numpy(np.stack([I.uniform_ising(b, 2 if chi == 4 else 1) for b in betas])).cuda()
    return torch.from_numpy(r.uniform(0.1, 1.1, (n, chi, chi, chi, chi))).cuda()


def _gemm_data(case, seed):
    g, t = _gen(seed), torch.float64 if case["dtype"] == "f64" else torch.float32
    shape = lambda rows: (case["batch"], rows, case["K"])  # noqa: E731
    return (torch.rand(shape(case["M"]), generator=g, device="cuda", dtype=torch.float64).to(t),
            torch.rand(shape(case["N"]), generator=g, device="cuda", dtype=torch.float64).to(t))


def prepare(case, seed):
    s, ctx = Held(case), _context()
    kind = case["kind"]
    if kind == "pass":
        s.net, s.data = _pass_data(case, seed)
        s.struct = pne.network_struct(s.net, data=s.data, n_batch=case["sets"])
        s.side, s.joined = torch.cuda.Stream(priority=-1), torch.cuda.Event()
    elif kind == "batch":
        s.parts, s.datas, terms = [], [], []
        for net, _, _, flat in _batch_data(case, seed):
            ns, keep = pne.network_struct(net, data=flat, n_batch=len(flat))
            part, _ = pne.pne_build_partition(ctx.h, ns, pne.PartitionOpts(1e-13, 10000, 0.0, 1))
            s.parts.append(s.own(pne.pne_partition_destroy, part))
            s.datas.append(flat)
            terms.append(s.own(pne.pne_terms_destroy,
                               pne.pne_enumerate_terms(ctx.h, part, pne.EnumOpts(case["K"], pne.PNE_MODE_LOOP, 1))[0]))
        s.batch = s.own(pne.pne_batch_destroy, pne.pne_batch_create(ctx.h, terms, DTYPES[case["dtype"]],
                                                                   pne.BatchOpts(4, 4, 1, pne.PNE_SCHED_HANDLE)))
        s.streams = [torch.cuda.Stream() for _ in range(8)]
    elif kind == "serve":
        s.requests = [(pne.network_struct(net, data=flat), K) for net, _, _, K, flat in _serve_data(case, seed)]
        s.server = s.own(pne.pne_server_destroy, pne.pne_server_create(
            ctx.h, pne.ServerOpts(64 << 30, 512, 12, 512, DTYPES[case["dtype"]], 0, 0)))
    elif kind == "comb":
        s.net = _lattice((3, 3), case["D"])
        s.data = _random_flat(sum(_site_sizes(s.net)), case["sets"], seed)
        s.struct = pne.network_struct(s.net, data=s.data, n_batch=case["sets"])
        s.lines = I.square3x3_six_lines()
    elif kind == "rank_r":
        nets, s.lines = _rank_r_data(case, seed)
        s.data = torch.from_numpy(np.concatenate([n.flat_data()[0] for n in nets])).cuda()
        s.struct = pne.network_struct(nets[0], data=s.data, n_batch=case["sets"])
    elif kind == "strip":
        s.A = _strip_data(case, seed)
    elif kind == "grid":
        s.net = _lattice((case["lx"], case["ly"]), case["chi"])
        s.data = _random_flat(sum(_site_sizes(s.net)), case["sets"], seed)
    else:
        s.A, s.B = _gemm_data(case, seed)
        s.C = torch.empty(case["batch"], case["M"], case["N"], dtype=s.A.dtype, device="cuda")
    return s


# ---------------------------------------------------------------- the calls
def _values(out):
    """The results' numbers as arrays: ln|Z| and the order sums, and the counts."""
    a = np.ctypeslib.as_array(out)
    orders = int(a["n_orders"].max())
    return {"log_abs": a["log_abs"].copy(), "sign": a["sign"].copy(), "c": a["c"][:, :orders].copy(),
            "n_terms": a["n_terms"].astype(np.int64), "n_clusters": a["n_clusters"].astype(np.int64)}


def _sum(ctx, terms, stream=None):
    out = (pne.Result * pne.pne_terms_n_results(terms))()
    if pne.load_library().pne_sum(ctx.h, terms, stream, out) != pne.PNE_OK:
        raise pne.PneError(-1, pne.pne_last_error(ctx.h))
    return _values(out)


def _run_pass(s):
    case, ctx = s.case, _context()
    main = torch.cuda.current_stream()
    apart = not case["cache"]      # recomputed: the search runs beside the sweeps, on a stream of its own
    side = s.side if apart else main
    part, _ = pne.pne_build_partition(ctx.h, s.struct[0], pne.PartitionOpts(1e-13, 10000, 0.0, case["arithmetic"],
                                                                             int(apart)), main.cuda_stream)
    try:
        terms, _, _ = pne.pne_enumerate_terms(ctx.h, part, pne.EnumOpts(case["K"], pne.PNE_MODE_LOOP,
                                                                         int(case["cache"])), side.cuda_stream)
        try:
            if apart:
                s.joined.record(side)
                main.wait_event(s.joined)
            pne.pne_contract_terms(ctx.h, terms, DTYPES[case["dtype"]], main.cuda_stream)
            return _sum(ctx, terms, main.cuda_stream)
        finally:
            pne.pne_terms_destroy(terms)
    finally:
        pne.pne_partition_destroy(part)


def _run_batch(s):
    ctx, main = _context(), torch.cuda.current_stream()
    for st in s.streams:
        st.wait_stream(main)
    opts = pne.PartitionOpts(1e-13, 10000, 0.0, 1, 1)
    for i, (part, data) in enumerate(zip(s.parts, s.datas)):
        pne.pne_partition_update(ctx.h, part, data, opts, s.streams[i % len(s.streams)].cuda_stream)
    for st in s.streams:
        main.wait_stream(st)
    out = (pne.Result * pne.pne_batch_n_results(s.batch))()
    if pne.load_library().pne_batch_run(ctx.h, s.batch, main.cuda_stream, out) != pne.PNE_OK:
        raise pne.PneError(-1, pne.pne_last_error(ctx.h))
    return _values(out)


def _run_serve(s):
    ids = [pne.pne_server_submit(s.server, ns[0], K) for ns, K in s.requests]
    pne.pne_server_drain(s.server)
    out = []
    for i in ids:
        status, r, _ = pne.pne_server_poll(s.server, i)
        if status != pne.PNE_OK:
            raise pne.PneError(status, pne.pne_server_first_error(s.server))
        out.append(r)
    return {"results": [np.concatenate([[r["log_abs"]], r["c"]]) for r in out],
            "counts": np.array([[r["n_terms"], r["n_clusters"]] for r in out])}


def _run_comb(s):
    ctx, stream = _context(), torch.cuda.current_stream().cuda_stream
    part, _ = pne.pne_build_partition(ctx.h, s.struct[0], pne.PartitionOpts(1e-13, 10000, 0.0, 1), stream)
    try:
        terms, _, _ = pne.pne_enumerate_combinatorial(ctx.h, part, s.lines, stream)
        try:
            pne.pne_contract_terms(ctx.h, terms, DTYPES[s.case["dtype"]], stream)
            return _sum(ctx, terms, stream)
        finally:
            pne.pne_terms_destroy(terms)
    finally:
        pne.pne_partition_destroy(part)


def _run_rank_r(s):
    case, ctx = s.case, _context()
    stream = torch.cuda.current_stream().cuda_stream
    w = pne.pne_weight_passing(ctx.h, s.struct[0], 0.8, 1e-10, 5000, stream)
    try:
        if case["dtype"] == "sitewise":
            res = pne.pne_rank_r_expand(ctx.h, w, case["rank"], case["form"], s.lines, case["sets"], stream)
        else:
            res = pne.pne_rank_r_expand_grid(ctx.h, w, case["rank"], case["form"], s.lines, case["sets"], 3, 3,
                                             DTYPES[case["dtype"]], stream)
    finally:
        pne.pne_weights_destroy(w)
    return {"log_abs": np.array([r["log_abs"] for r in res]), "n_terms": np.array([r["n_terms"] for r in res])}


def _run_strip(s):
    case = s.case
    res = pne.pne_strip_expansion(_context().h, s.A, case["L"], True, arithmetic=case["arithmetic"],
                                  stream=torch.cuda.current_stream().cuda_stream)
    return {"f": np.array([r["f"] for r in res]), "log_lam": np.array([r["log_lam"][1:] for r in res]),
            "log_gam": np.array([r["log_gam"][1:] for r in res]),
            "log_z": np.array([[row[1:] for row in r["log_z"][1:]] for r in res])}


def _run_grid(s):
    case = s.case
    res = pne.pne_grid_contract(_context().h, s.net, case["lx"], case["ly"], DTYPES[case["dtype"]], data=s.data,
                                n_batch=case["sets"], stream=torch.cuda.current_stream().cuda_stream)
    return {"log_abs": np.array([r["log_abs"] for r in res]), "sign": np.array([r["sign"] for r in res])}


def _run_gemm(s):
    pne.pne_dense_gemm(_context().h, DTYPES[s.case["dtype"]], s.A, s.B, s.C, torch.cuda.current_stream().cuda_stream)
    return s.C


def run(state):
    return {"pass": _run_pass, "batch": _run_batch, "serve": _run_serve, "comb": _run_comb, "rank_r": _run_rank_r,
            "strip": _run_strip, "grid": _run_grid, "gemm": _run_gemm}[state.case["kind"]](state)


# ---------------------------------------------------------------- what a pass cannot do without
def _expansion_work(shape, D, sets, K):
    """Tensors in, results out; 30 sweeps of one multiply-add per entry and leg, the gauge transform of every leg,
    and a few operations per term."""
    net = _lattice(shape, D)
    sizes, legs = _site_sizes(net), np.diff(net.site_ptr)
    entries = float(np.dot(sizes, legs))
    growth = {2: (1.0, 2.6), 3: (3.0, 5.5)}[len(shape)]
    clusters = math.prod(shape) * sum(growth[0] * growth[1] ** (k - 4) / 2 for k in range(4, min(K, 10) + 1))
    return {"bytes": sets * (8.0 * sum(sizes) + 8.0 * (K + 4)),
            "flops": sets * (2.0 * entries * (30 + D) + 4.0 * clusters * K * (D - 1) ** 2)}


def _added(works):
    works = list(works)
    return {k: sum(w[k] for w in works) for k in ("bytes", "flops")}


def work(case):
    kind = case["kind"]
    if kind == "pass":
        return _expansion_work(_shape(case), case["D"], case["sets"], case["K"])
    if kind == "batch":
        return _added(_expansion_work((L, L), D, len(kinds), case["K"]) for (L, D), kinds in _batch_groups(case))
    if kind == "serve":
        return _added(_expansion_work(shape, D, 1, K) for _, shape, D, K, _ in _serve_data(case, 0))
    if kind == "comb":
        w = _expansion_work((3, 3), case["D"], case["sets"], 4)
        return {"bytes": w["bytes"], "flops": w["flops"] + case["sets"] * 63 * 9 * 2.0 * case["D"] ** 5}
    if kind == "rank_r":
        d, n = 2 ** case["block"], case["sets"]
        entries = 4 * d ** 2 + 4 * d ** 3 + d ** 4
        terms = 63 if case["form"] else 4
        # 30 sweeps; an update reduces both tensors to triangles and multiplies the leg of each
        return {"bytes": 8.0 * n * entries, "flops": n * (30 * 4.0 * d * (8 * d ** 2 + 12 * d ** 3 + 4 * d ** 4)
                                                          + terms * 9 * 2.0 * d ** 3 * case["rank"] ** 2)}
    if kind == "strip":
        chi, L, n = case["chi"], case["L"], case["sets"]
        rows = sum(2.0 * chi ** (k + 2) * (2 + max(0, k - 2) * chi) for k in range(1, L + 1))
        return {"bytes": n * 8.0 * (chi ** 4 + L * L + 2 * L + 1), "flops": n * 2 * 20 * rows}
    if kind == "grid":
        lx, ly, chi, n = case["lx"], case["ly"], case["chi"], case["sets"]
        flops, cut = 0.0, 1.0
        for y in range(ly):
            for x in range(lx):
                up, left = chi ** (y > 0), chi ** (x > 0)
                down, right = chi ** (y < ly - 1), chi ** (x < lx - 1)
                flops += 2.0 * cut * down * right
                cut = cut / (up * left) * down * right
        return {"bytes": 8.0 * n * sum(_site_sizes(_lattice((lx, ly), chi))), "flops": n * flops}
    b, M, N, K = case["batch"], case["M"], case["N"], case["K"]
    return {"bytes": (8.0 if case["dtype"] == "f64" else 4.0) * b * (M * K + N * K + M * N),
            "flops": 2.0 * b * M * N * K}


# ---------------------------------------------------------------- the same in 64 bits
@functools.lru_cache(maxsize=None)
def _loop_shapes(dim, K):
    """Connected bond sets of at most K <= 8 bonds without loose ends on the infinite lattice, one per translation:
    closed walks and paths between two sites of a smaller set, added to it (two rings joined by a path need nine)."""
    steps = [tuple(int(i == a) * sg for i in range(dim)) for a in range(dim) for sg in (1, -1)]
    add = lambda p, q: tuple(x + y for x, y in zip(p, q))  # noqa: E731

    def canon(edges):
        low = [min(min(a[i], b[i]) for a, b in edges) for i in range(dim)]
        sub = lambda p: tuple(x - y for x, y in zip(p, low))  # noqa: E731
        return frozenset((sub(a), sub(b)) for a, b in edges)

    def ears(sites, edges, most):
        def walk(start, at, path, seen):
            for st in steps:
                to = add(at, st)
                e = (min(at, to), max(at, to))
                if e in edges or e in path:
                    continue
                if to in sites:
                    yield path + [e]
                elif to not in seen and len(path) + 1 < most and \
                        min(sum(abs(x - y) for x, y in zip(to, v)) for v in sites) <= most - len(path) - 1:
                    yield from walk(start, to, path + [e], seen | {to})
        for v in sites:
            yield from walk(v, v, [], frozenset())

    origin = (0,) * dim
    found = {canon(p) for p in ears({origin}, frozenset(), K)}
    new = set(found)
    while new:
        grown = set()
        for edges in new:
            if len(edges) < K:
                sites = {v for e in edges for v in e}
                grown |= {canon(edges | set(p)) for p in ears(sites, edges, K - len(edges))}
        new = grown - found
        found |= new
    return sorted((sorted(e) for e in found), key=lambda e: (len(e), e))


class _Lattice64:
    """Site tensors [sets, sites] with 2 dim legs each (down the axes z, y, x, then up x, y, z, the order of their
    bonds' numbers); a leg that leaves the lattice holds its first value only."""

    def __init__(self, shape, D, flat):
        self.shape, self.D, self.dim = shape, D, len(shape)
        self.sets, N = flat.shape[0], int(np.prod(shape))
        self.axes = list(range(self.dim))[::-1] + list(range(self.dim))
        self.sign = [-1] * self.dim + [1] * self.dim
        n = 2 * self.dim
        self.T = torch.zeros((self.sets, N) + (D,) * n, dtype=torch.float64, device=flat.device)
        self.pos = [tuple(int(v // np.prod(shape[:i], dtype=int)) % shape[i] for i in range(self.dim)) for v in range(N)]
        self.at = {p: v for v, p in enumerate(self.pos)}
        self.near, off = [], 0
        for v, p in enumerate(self.pos):
            near = []
            for a, sg in zip(self.axes, self.sign):
                q = list(p)
                q[a] += sg
                near.append(self.at.get(tuple(q), -1))
            legs = [i for i in range(n) if near[i] >= 0]
            size = D ** len(legs)
            where = tuple(slice(None) if i in legs else 0 for i in range(n))
            self.T[(slice(None), v) + where] = flat[:, off:off + size].reshape((self.sets,) + (D,) * len(legs))
            off += size
            self.near.append(near)
        self.near = torch.tensor(self.near, device=flat.device)
        self.opposite = list(range(n))[::-1]
        self._messages()
        self._blocks = {}

    def _cap(self, T, m, keep):
        """T with every leg but those kept contracted with the messages arriving on it."""
        n = 2 * self.dim
        for i in reversed(range(n)):
            if i not in keep:
                after = sum(1 for j in keep if j > i)
                T = torch.einsum("svxab,sva->svxb", T.reshape(T.shape[0], T.shape[1], -1, self.D, self.D ** after),
                                 m[:, :, i])
        return T.reshape((T.shape[0], T.shape[1]) + (self.D,) * len(keep))

    def _messages(self):
        n, D = 2 * self.dim, self.D
        start = torch.full((self.sets, len(self.pos), n, D), D ** -0.5, dtype=torch.float64, device=self.T.device)
        edge = torch.zeros(D, dtype=torch.float64, device=self.T.device)
        edge[0] = 1.0
        inside = (self.near >= 0)[None, :, :, None]
        arriving = lambda out: torch.where(inside, torch.stack(  # noqa: E731
            [out[:, self.near[:, i], self.opposite[i]] for i in range(n)], 2), edge)
        m, settled = arriving(start), 0.0
        for _ in range(2000):
            out = torch.stack([self._cap(self.T, m, [i]) for i in range(n)], 2)
            out = out / out.norm(dim=-1, keepdim=True)
            big = out.gather(-1, out.abs().argmax(-1, keepdim=True))
            new = arriving(out * torch.sign(big))
            change = float((new - m).abs().max())
            m = new
            if change < 1e-14 or (settled and change > 0.5 * settled):
                break
            settled = change if change < 1e-12 else 0.0
        self.m = m
        self.z = self._cap(self.T, m, [])
        # overlap of the two messages of a bond, seen from either end
        far = torch.where(inside, torch.stack([m[:, self.near[:, i], self.opposite[i]] for i in range(n)], 2), edge)
        self.n = (m * far).sum(-1)

    def block(self, legs):
        """Site tensors over the given legs, the others capped, divided by the fully capped value; Q = 1 - P and the
        overlap of every bond towards a higher site go into that site's lower end."""
        if legs not in self._blocks:
            B = self._cap(self.T, self.m, list(legs)) / self.z.reshape(self.z.shape + (1,) * len(legs))
            for k, i in enumerate(legs):
                if self.sign[i] > 0:
                    far = self.m[:, self.near[:, i], self.opposite[i]]
                    n = self.n[:, :, i]
                    P = torch.einsum("sva,svb->svab", self.m[:, :, i], far) / n[:, :, None, None]
                    Q = (torch.eye(self.D, dtype=torch.float64, device=B.device) - P) * n[:, :, None, None]
                    B = torch.einsum("svxab,svac->svxcb", B.reshape(self.sets, B.shape[1], -1, self.D,
                                                                    self.D ** (len(legs) - 1 - k)), Q)
            self._blocks[legs] = B.reshape((self.sets, -1) + (self.D,) * len(legs))
        return self._blocks[legs]

    def clusters(self, K):
        """{size: [(values [sets, placements], sites [placements, sites of one])]} of every set in _loop_shapes."""
        found = {}
        for edges in _loop_shapes(self.dim, K):
            sites = sorted({v for e in edges for v in e})
            top = [max(v[i] for v in sites) for i in range(self.dim)]
            if any(t >= s for t, s in zip(top, self.shape)):
                continue
            anchors = [p for p in itertools.product(*(range(s - t) for s, t in zip(self.shape, top)))]
            at = torch.tensor([[self.at[tuple(a + b for a, b in zip(p, v))] for v in sites] for p in anchors],
                              device=self.T.device)
            order, seen = [sites[0]], {sites[0]}
            while len(order) < len(sites):       # along the bonds, so that few legs are open at a time
                order.append(next(w for v in reversed(order) for e in edges if v in e for w in e if w not in seen))
                seen.add(order[-1])
            total, open_ = None, ""
            for v in order:
                legs, names = [], ""
                for i, (a, sg) in enumerate(zip(self.axes, self.sign)):
                    w = tuple(x + sg * (j == a) for j, x in enumerate(v))
                    if (min(v, w), max(v, w)) in edges:
                        legs.append(i)
                        names += chr(99 + edges.index((min(v, w), max(v, w))))
                B = self.block(tuple(legs))[:, at[:, sites.index(v)]]
                if total is None:
                    total, open_ = B, names
                else:
                    rest = "".join(c for c in open_ if c not in names) + "".join(c for c in names if c not in open_)
                    total, open_ = torch.einsum(f"ab{open_},ab{names}->ab{rest}", total, B), rest
            found.setdefault(len(edges), []).append((total, at))
        return found

    def expansion(self, K):
        """ln|Z_K| and the order sums; K <= 8: a term holds two clusters only where both have four bonds."""
        c = torch.zeros(self.sets, K + 1, dtype=torch.float64, device=self.T.device)
        c[:, 0] = 1.0
        found = self.clusters(K)
        for k, groups in found.items():
            c[:, k] += sum(w.sum(1) for w, _ in groups)
        if K == 8 and 4 in found:
            w = torch.cat([w for w, _ in found[4]], 1)
            sites = torch.cat([a for _, a in found[4]], 0)
            on = torch.zeros(len(sites), len(self.pos), dtype=torch.float64, device=w.device).scatter_(1, sites, 1.0)
            apart = (on @ on.T == 0).to(torch.float64)
            c[:, 8] += 0.5 * torch.einsum("si,ij,sj->s", w, apart, w)
        log_abs = self.log_reference() + c.sum(1).abs().log()
        return {"log_abs": log_abs.cpu().numpy(), "c": c.cpu().numpy()}

    def log_reference(self):
        """ln of the network with every bond capped."""
        return self.z.abs().log().sum(1) - self.n[:, :, self.dim:].abs().log().sum((1, 2))


def _ising_full_order(case, seed):
    """Even bond subsets of a small lattice, counted by size over its cycle space: c_k = N_k tanh(beta)^k."""
    net = _lattice(_shape(case), 2)
    M, N = net.n_bonds, net.n_sites
    lx, ly = _shape(case)
    number = {(int(a), int(b)): i for i, (a, b) in enumerate(net.bond_site)}
    counts, masks = np.zeros(M + 1, dtype=np.int64), np.zeros(1, dtype=np.int64)
    for y in range(ly - 1):
        for x in range(lx - 1):
            s = y * lx + x
            ring = sum(1 << number[e] for e in ((s, s + 1), (s, s + lx), (s + 1, s + lx + 1), (s + lx, s + lx + 1)))
            masks = np.concatenate([masks, masks ^ ring])
    for m in masks.tolist():
        counts[bin(m).count("1")] += 1
    betas = _betas(case, seed, case["sets"])
    c = np.stack([counts[:case["K"] + 1] * math.tanh(b) ** np.arange(case["K"] + 1.0) for b in betas])
    return {"log_abs": np.array([N * math.log(2) + M * math.log(math.cosh(b)) for b in betas]) + np.log(c.sum(1)),
            "c": c}


def _contract_grid(lx, ly, site):
    """A grid's value per set, ln and sign: site(x, y) gives [sets, up, left, right, down]; row by row."""
    W, log = None, 0.0
    for y in range(ly):
        for x in range(lx):
            T = site(x, y)
            n, up, left, right, down = T.shape
            if W is None:
                W = T.new_ones(n, 1, 1, 1)
            # W [sets, legs of this row already made, left, legs of the row above still open]; up comes first of those
            W = W.reshape(n, -1, left, up, W.shape[3] // up)
            W = torch.matmul(W.permute(0, 1, 4, 3, 2).reshape(n, -1, up * left), T.reshape(n, up * left, right * down)) \
                .reshape(n, W.shape[1], W.shape[4], right, down).permute(0, 1, 4, 3, 2).reshape(n, -1, right, W.shape[4])
            top = W.abs().amax((1, 2, 3), keepdim=True)
            W, log = W / top, log + top.reshape(n).log()
        W = W.reshape(W.shape[0], 1, 1, -1)
    W = W.reshape(-1)
    return log + W.abs().log(), torch.sign(W)


def _exact_grid_case(case, seed):
    lx, ly, chi = case["lx"], case["ly"], case["chi"]
    flat = _random_flat(sum(_site_sizes(_lattice((lx, ly), chi))), case["sets"], seed)
    off = 0
    tensors = {}
    for y in range(ly):
        for x in range(lx):
            legs = [chi ** (y > 0), chi ** (x > 0), chi ** (x < lx - 1), chi ** (y < ly - 1)]
            tensors[x, y] = flat[:, off:off + math.prod(legs)].reshape([-1] + legs)
            off += math.prod(legs)
    log, sign = _contract_grid(lx, ly, lambda x, y: tensors[x, y])
    return {"log_abs": log.cpu().numpy()}


def _six_lines():
    """The lines between the columns, between the rows and across the corner of a 3 x 3 lattice: the bonds
    (lower site, axis) each cuts."""
    lines = [{((x, y), 0) for y in range(3)} for x in (0, 1)] + [{((x, y), 1) for x in range(3)} for y in (0, 1)]
    return lines + [{((x, k - x), a) for x in range(3) for a in (0, 1) if 0 <= k - x < 3 and (x, k - x)[a] < 2}
                    for k in (0, 1)]


def _exact_comb(case, seed):
    D, n = case["D"], case["sets"]
    lat = _Lattice64((3, 3), D, _random_flat(sum(_site_sizes(_lattice((3, 3), D))), n, seed))
    edge = lambda v, i: D if lat.near[v, i] >= 0 else 1  # noqa: E731
    lines, ref = _six_lines(), lat.log_reference()
    c = torch.zeros(n, 7, dtype=torch.float64, device=ref.device)
    for size in range(1, 7):
        for x in itertools.combinations(lines, size):
            cut = set().union(*x)

            def site(px, py):
                v = py * 3 + px
                T = lat.T[:, v]
                for i, a in ((2, 0), (3, 1)):
                    if ((px, py), a) in cut:
                        w = lat.near[v, i]
                        P = torch.einsum("sa,sb->sab", lat.m[:, v, i], lat.m[:, w, lat.opposite[i]]) \
                            / lat.n[:, v, i, None, None]
                        T = torch.einsum("suled,sea->sulad" if i == 2 else "sulre,sea->sulra", T, P)
                return T[:, :edge(v, 0), :edge(v, 1), :edge(v, 2), :edge(v, 3)]
            log, sign = _contract_grid(3, 3, site)
            c[:, size] += sign * torch.exp(log - ref)
    total = sum((-1) ** (k + 1) * c[:, k] for k in range(1, 7))
    return {"log_abs": (ref + total.abs().log()).cpu().numpy(), "c": c.cpu().numpy()}


def _weighted(net, alpha, tol):
    """Weight passing on one network: the tensors with the weights' roots on every leg, and the log of the scale."""
    T = [np.asarray(t, dtype=np.float64) for t in net.tensors]
    S = [np.ones(int(d)) for d in net.bond_dim]
    legs = [[int(b) for b in net.legs(v)] for v in range(net.n_sites)]

    def triangle(v, bond):
        t = T[v]
        for i, b in enumerate(legs[v]):
            if b != bond:
                t = t * S[b].reshape([-1 if j == i else 1 for j in range(t.ndim)])
        t = np.moveaxis(t, legs[v].index(bond), -1)
        _, s, vt = np.linalg.svd(np.linalg.qr(t.reshape(-1, t.shape[-1]), mode="r"))
        return s, vt

    def on_leg(v, bond, X):
        i = legs[v].index(bond)
        T[v] = np.moveaxis(np.tensordot(T[v], X, axes=([i], [0])), -1, i)
    scale = 0.0
    for _ in range(5000):
        change = 0.0
        for b, (u, v) in enumerate(net.bond_site):
            sa, vat = triangle(int(u), b)
            sb, vbt = triangle(int(v), b)
            uc, sc, vct = np.linalg.svd((sa[:, None] * vat) @ (S[b][:, None] * vbt.T) * sb)
            g = sc ** ((1 - alpha) / 2)
            on_leg(int(u), b, vat.T @ (uc / sa[:, None]) * g)
            on_leg(int(v), b, vbt.T @ (vct.T / sb[:, None]) * g)
            new = sc ** alpha
            scale += math.log(new[0])
            change = max(change, float(np.abs(new / new[0] - S[b]).max()))
            S[b] = new / new[0]
        if change < tol:
            break
    for v in range(net.n_sites):
        for b in legs[v]:
            on_leg(v, b, np.diag(np.sqrt(S[b])))
    return T, scale


def _exact_rank_r(case, seed):
    nets, parts = _rank_r_data(case, seed)
    r, M, out = case["rank"], len(parts), []
    if case["form"]:
        terms = [((-1) ** (len(x) + 1), {b: slice(0, r) for p in x for b in parts[p]})
                 for k in range(1, M + 1) for x in itertools.combinations(range(M), k)]
    else:
        terms = [(1, {**{parts[p][0]: slice(r, None) for p in range(k)}, parts[k][0]: slice(0, r)}) for k in range(M)]
    for net in nets:
        T, scale = _weighted(net, 0.8, 1e-12)
        T = [torch.from_numpy(t).cuda() for t in T]
        total = 0.0
        for sg, kept in terms:
            def site(x, y):
                v = y * 3 + x
                t = T[v][tuple(kept.get(int(b), slice(None)) for b in net.legs(v))]
                dims, inside = iter(t.shape), (y > 0, x > 0, x < 2, y < 2)
                return t.reshape([1] + [next(dims) if has else 1 for has in inside])
            log, sign = _contract_grid(3, 3, site)
            total += sg * float(sign * torch.exp(log))
        out.append(scale + math.log(abs(total)))
    return {"log_abs": np.array(out)}


def _strip_side(A, m, L):
    """ln of the leading eigenvalue of a row of k sites, and of the capped patches of 1..L rows, for k = 1..L."""
    mR, mL, mD, mU = m
    n, chi = A.shape[0], A.shape[1]
    lam, patches = [], []
    for k in range(1, L + 1):
        v = functools.reduce(lambda a, b: torch.einsum("np,nu->npu", a, b).reshape(n, -1), [mD] * k)
        close = functools.reduce(lambda a, b: torch.einsum("np,nu->npu", a, b).reshape(n, -1), [mU] * k)
        log, rows, last = torch.zeros(n, dtype=A.dtype, device=A.device), [], None
        for it in range(400):
            before = (v * v).sum(1)
            W = torch.einsum("nh,np->nhp", mR, v)
            for j in range(k):
                W = torch.einsum("nhpus,nhurd->nrpds", W.reshape(n, chi, chi ** j, chi, -1), A)
            W = torch.einsum("nh,nhp->np", mL, W.reshape(n, chi, -1))
            estimate = ((v * W).sum(1) / before).log()
            top = W.abs().amax(1)
            v, log = W / top[:, None], log + top.log()
            if len(rows) < L:
                rows.append(log + (v * close).sum(1).log())
            if last is not None and it >= L and float((estimate - last).abs().max()) < 1e-15:
                break
            last = estimate
        lam.append(estimate)
        patches.append(torch.stack(rows, 1))
    return torch.stack(lam, 1), torch.stack(patches, 1)


def _exact_strip(case, seed):
    A, L = _strip_data(case, seed), case["L"]
    n, chi = A.shape[0], A.shape[1]
    m = [torch.full((n, chi), chi ** -0.5, dtype=A.dtype, device=A.device) for _ in range(4)]
    for _ in range(20000):
        mR, mL, mD, mU = m
        new = [torch.einsum(e, A, a, b, c) for e, a, b, c in (
            ("nlurd,nl,nu,nd->nr", mR, mD, mU), ("nlurd,nr,nu,nd->nl", mL, mD, mU),
            ("nlurd,nl,nr,nu->nd", mR, mL, mD), ("nlurd,nl,nr,nd->nu", mR, mL, mU))]
        new = [x / x.norm(dim=1, keepdim=True) for x in new]
        change = max(float((a - b).abs().max()) for a, b in zip(new, m))
        m = new
        if change < 1e-15:
            break
    h, w = (m[0] * m[1]).sum(1, keepdim=True).sqrt(), (m[2] * m[3]).sum(1, keepdim=True).sqrt()
    m = [m[0] / h, m[1] / h, m[2] / w, m[3] / w]
    lam, z = _strip_side(A, m, L)
    gam, _ = _strip_side(A.permute(0, 2, 1, 4, 3).contiguous(), [m[2], m[3], m[0], m[1]], L)
    ref = torch.einsum("nlurd,nl,nu,nr,nd->n", A, m[0], m[2], m[1], m[3]).log().cpu().numpy()
    lam, gam, z = lam.cpu().numpy(), gam.cpu().numpy(), z.cpu().numpy()
    gaps, signs = np.zeros((1 << L, L)), np.ones(1 << L)
    for mask in range(1, 1 << L):
        cuts = [i for i in range(L) if mask >> i & 1]
        for a, b in zip(cuts, cuts[1:] + [cuts[0] + L]):
            gaps[mask, b - a - 1] += 1
        signs[mask] = (-1) ** len(cuts)
    f = []
    for i in range(n):
        t = gaps @ z[i] @ gaps.T
        t[0, :], t[:, 0] = L * (gaps @ gam[i]), L * (gaps @ lam[i])
        terms = -np.outer(signs, signs) * np.expm1(t - L * L * ref[i])
        terms[0, 0] = 0.0
        # the signs of all terms but the empty one sum to one
        f.append(-(L * L * ref[i] + math.log1p(math.fsum(terms.ravel().tolist()))) / (L * L))
    return {"f": np.array(f), "log_lam": lam, "log_gam": gam, "log_z": z}


def exact(case, seed):
    kind = case["kind"]
    if kind == "gemm":
        A, B = _gemm_data(case, seed)
        return torch.matmul(A.double(), B.double().transpose(1, 2))
    if kind == "grid":
        return _exact_grid_case(case, seed)
    if kind == "comb":
        return _exact_comb(case, seed)
    if kind == "strip":
        return _exact_strip(case, seed)
    if kind == "rank_r":
        return _exact_rank_r(case, seed)
    if kind == "pass":
        if case["K"] > 8:
            return _ising_full_order(case, seed) if case["shape"] == "4x4" and case["K"] == 24 else None
        _, flat = _pass_data(case, seed)
        return _Lattice64(_shape(case), case["D"], flat).expansion(case["K"])
    if kind == "batch":
        each = [_Lattice64(shape, D, flat).expansion(case["K"]) for _, shape, D, flat in _batch_data(case, seed)]
        return {k: np.concatenate([e[k] for e in each]) for k in ("log_abs", "c")}
    out = []
    for _, shape, D, K, flat in _serve_data(case, seed):
        if len(shape) == 3 and (K > 7 or D ** 6 * math.prod(shape) > 2e6):
            out.append(None)      # thousands of cluster shapes, or tensors too large to do quickly
            continue
        e = _Lattice64(shape, D, torch.from_numpy(flat)[None].cuda()).expansion(K)
        out.append(np.concatenate([e["log_abs"], e["c"][0]]))
    return {"results": out}
