"""The work that a user of this package has it do, as measurable cases.

A user trains a vector of parameters with evolution strategies: the parameters are split
into subspaces, each visit of a subspace perturbs it once per population member, restores
it, shapes the members' rewards and applies the update.  The cases are whole visits and
steps through the schedules (``es``) over the range of model sizes, populations, working
copies and subspace kinds the repository configures, the partition build, and single calls
(``copes``) as a program with its own schedule makes them, odd and ragged sizes among them.

Case kinds:
  visit      es.round_robin_visit on one subspace
  sync       es.sync_step (Algorithm 1) on random chunks resampled every step
  backup     es.backup_visit, the context in pinned host memory
  partition  copes_hash_count + copes_hash_fill: a hash partition as index lists
  call       one perturb / pair / two_pairs / update / init call
"""
import ctypes
import math

import numpy as np
import torch

from paper_2608_02391_gb300 import copes, es, workloads

SIGMA, ALPHA, BASE_SEED, PARTITION_SEED, ITERATION = 1e-3, 5e-4, 33, 1088, 2
NAMED = ("4b", "0.5b", "4b-hash-slice")  # layouts of workloads.workload()


# ------------------------------------------------------------------------------- cases
def listed():
    return [
        # the smallest visit: one fp32 vector of 2^20, K = 4, N = 8 (launch and host latency)
        _visit("visit-tiny-fp32", layout="vector", n=1 << 20, K=4, k=1, N=8, dtype="fp32", copies=1),
        # a small model's layer block, four working copies, centred ranks
        _visit("visit-0.5b", layout="0.5b", K=8, k=1, mode="groups", N=16, copies=4, shaping="centered_rank"),
        # the 4B model's layer block, N = 32, four working copies (the benchmark's visit)
        _visit("visit-4b", layout="4b", K=8, k=1, mode="groups", N=32, copies=4),
        # the 8B model's lm_head as its own subspace, N = 128 (64 noise vectors), two copies
        _visit("visit-8b-head", layout="vector", n=4096 * 151936, K=1, k=0, N=128, copies=2, sigma=5e-4),
        # an odd-sized vector cut at odd places, small tiles, one-sided population of 7
        _visit("visit-ragged", layout="vector", n=33_333_337, K=3, k=1, N=7, copies=1, pairing="one_sided",
               tile=1000, shaping="none"),
        # Algorithm 1 on the 4B model: the partition is resampled every step
        _sync("sync-4b", layout="4b", K=4, N=32, copies=2),
        # hash subspaces (1 element in 16): index lists with a gathered master, and replayed
        # from the seed with a per-visit membership mask
        _visit("visit-hash-gathered", layout="4b-hash-slice", K=16, k=3, mode="hash-gathered", N=64, copies=2),
        _visit("visit-hash-mask", layout="4b-hash-slice", K=16, k=3, mode="hash-mask", N=64, copies=2),
        # the context in pinned host memory (a GPU with no room for an fp32 master)
        {"name": "visit-backup", "kind": "backup", "n": 1 << 27, "K": 2, "k": 1, "N": 16, "tile": 16384},
        # the hash partition of a small model as index lists
        {"name": "partition-hash-0.5b", "kind": "partition", "layout": "0.5b", "n": 0, "K": 16},
        # a program with its own schedule: one antithetic pair of a mid-sized block, and one
        # update of a small block from many noise vectors
        {"name": "call-pair-odd", "kind": "call", "op": "pair", "n": 14_909_441, "begin": 36, "end": 14_909_441,
         "tile": 16384, "dtype": "bf16", "N": 2},
        {"name": "call-update-small", "kind": "call", "op": "update", "n": 1 << 20, "begin": 0, "end": 1 << 20,
         "tile": 16384, "dtype": "bf16", "N": 64},
    ]


def _visit(name, layout, K, k, N, n=0, mode="contiguous", dtype="bf16", copies=1, sigma=SIGMA, shaping="zscore",
           pairing="antithetic", tile=16384):
    return {"name": name, "kind": "visit", "layout": layout, "n": n, "K": K, "k": k, "mode": mode, "N": N,
            "dtype": dtype, "copies": copies, "sigma": sigma, "shaping": shaping, "pairing": pairing, "tile": tile}


def _sync(name, layout, K, N, copies, n=0, chunk=65536):
    return {"name": name, "kind": "sync", "layout": layout, "n": n, "K": K, "N": N, "copies": copies, "chunk": chunk}


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: sizes over their logarithm, odd ones among them; the noise generated
    (elements x noise vectors) stays below the largest listed case's."""
    kind = rng.choice(["visit", "visit", "visit", "hash", "sync", "backup", "partition", "call", "call", "call"])
    if kind == "visit":
        n, K = _log_int(rng, 40_000, 600_000_000), rng.choice([1, 2, 3, 4, 7, 8])
        pairing = rng.choice(["antithetic", "antithetic", "one_sided"])
        N = 2 * _log_int(rng, 1, 64) if pairing == "antithetic" else _log_int(rng, 1, 32)
        if n // K * N > 10_000_000_000:
            N = max(2, 10_000_000_000 // (n // K) // 2 * 2)
        return _unnamed(_visit("", layout="vector", n=n, K=K, k=rng.randrange(K), N=N,
                               dtype=rng.choice(["bf16", "bf16", "fp32"]), copies=rng.choice([1, 2, 4]),
                               shaping=rng.choice(["zscore", "centered_rank", "none"]), pairing=pairing,
                               tile=rng.choice([16384, 16384, 16384, 4096, 65536, 1000])))
    if kind == "hash":
        K = rng.choice([2, 4, 16, 64])
        return _unnamed(_visit("", layout="vector", n=_log_int(rng, 100_000, 200_000_000), K=K, k=rng.randrange(K),
                               mode=rng.choice(["hash-lists", "hash-gathered", "hash-mask", "hash-replay"]),
                               N=2 * _log_int(rng, 1, 16), copies=rng.choice([1, 2]),
                               dtype=rng.choice(["bf16", "bf16", "fp32"])))
    if kind == "sync":
        K = rng.choice([2, 4, 8])
        return _unnamed(_sync("", layout="vector", n=_log_int(rng, 4_000_000, 1_000_000_000), K=K,
                              N=2 * K * rng.randrange(1, 5), copies=rng.choice([1, 2, 4])))
    if kind == "backup":
        return {"kind": "backup", "n": _log_int(rng, 100_000, 1 << 27), "K": 2, "k": rng.randrange(2),
                "N": 2 * _log_int(rng, 1, 16), "tile": 16384}
    if kind == "partition":
        return {"kind": "partition", "layout": "vector", "n": _log_int(rng, 100_000, 500_000_000),
                "K": rng.choice([2, 4, 7, 16, 64])}
    n = _log_int(rng, 20_000, 600_000_000)
    begin = rng.randrange(0, n // 8)
    if rng.random() < 0.5:
        begin &= ~63
    op = rng.choice(["perturb", "pair", "two_pairs", "update", "update", "init"])
    return {"kind": "call", "op": op, "n": n, "begin": begin, "end": n - rng.randrange(0, n // 8),
            "tile": rng.choice([16384, 16384, 16384, 4096, 65536, 1000]), "dtype": rng.choice(["bf16", "bf16", "fp32"]),
            "N": 2 * _log_int(rng, 1, 32) if op == "update" else 2}


def _unnamed(case):
    del case["name"]
    return case


# ------------------------------------------------------------------------------- inputs
def _numel(case):
    if case.get("layout") in NAMED:
        return workloads.workload(case["layout"]).numel
    return [case["n"]]


def _span(case):
    """[begin, end) of a contiguous or layer-group subspace as global ranges."""
    numel = _numel(case)
    if case["mode"] == "groups":
        wl = workloads.workload(case["layout"])
        off = workloads.layout_offsets(wl.tensors)
        return [(off[t], off[t] + m) for t, m in enumerate(numel) if wl.group_of[t] == case["k"]]
    n = numel[0]
    return [(n * case["k"] // case["K"], n * (case["k"] + 1) // case["K"])]


def _d_k(case):
    """Elements the case's subspace holds (hash: the expected count)."""
    if case["kind"] == "call":
        return case["end"] - case["begin"]
    if case["kind"] in ("sync", "partition") or case.get("mode", "").startswith("hash"):
        return sum(_numel(case)) // (1 if case["kind"] in ("sync", "partition") else case["K"])
    if case["kind"] == "backup":
        return case["n"] * (case["k"] + 1) // case["K"] - case["n"] * case["k"] // case["K"]
    return sum(e - b for b, e in _span(case))


def _theta(n, seed, dtype=torch.float32):
    """Weights as a trained model's: N(0, 0.02^2)."""
    gen = torch.Generator("cuda").manual_seed(seed)
    return torch.randn(n, generator=gen, device="cuda", dtype=dtype).mul_(0.02)


def _rewards(n, seed):
    """Mean of 16 verifier outcomes per member, as the benchmark's."""
    rng = np.random.Generator(np.random.PCG64(seed))
    return workloads.bernoulli_rewards(rng, n, 16, 0.2, 0.6)


def _fitness(n, seed):
    return np.random.Generator(np.random.PCG64(seed)).standard_normal(n).astype(np.float32)


_DTYPE = {"bf16": torch.bfloat16, "fp32": torch.float32}


def _arena(n, seed, dtype, copies):
    master = _theta(n, seed)
    w = [master.to(_DTYPE[dtype]) if dtype == "bf16" else master.clone()]
    w += [w[0].clone() for _ in range(copies - 1)]
    return copes.Arena(w[0], master, *w[1:])


def _config(case):
    if case["kind"] == "sync":
        return es.ESConfig(case["N"], SIGMA, ALPHA, convention=copes.COEF_PAPER, dimension_aware=True,
                           base_seed=BASE_SEED)
    return es.ESConfig(case["N"], case.get("sigma", SIGMA), ALPHA, shaping=case.get("shaping", "zscore"),
                       pairing=copes.ONE_SIDED if case.get("pairing") == "one_sided" else copes.ANTITHETIC,
                       base_seed=BASE_SEED)


def _partner(arena, copies):
    return {1: lambda: None, 2: lambda: es.Partner.second_copy(arena), 4: lambda: es.Partner.four_copies(arena)}[copies]()


def prepare(case, seed):
    kind = case["kind"]
    if kind == "call":
        copies = {"pair": 2, "two_pairs": 4}.get(case["op"], 1)
        arena = _arena(case["n"], seed, case["dtype"], copies)
        nid, sign, P = copes.member_table(case["N"], copes.ANTITHETIC)
        return {"case": case, "arena": arena, "nid": nid, "sign": sign,
                "sub": copes.tiles_from_ranges([(case["begin"], case["end"])], tile_size=case["tile"]),
                "seeds": copes.member_seeds(BASE_SEED, ITERATION, 0, max(P, 2)),
                "fitness": torch.from_numpy(_fitness(case["N"], seed)).cuda()}
    if kind == "partition":
        return _prepare_partition(case, seed)
    if kind == "backup":
        w = _theta(case["n"], seed).to(torch.bfloat16)
        arena = copes.BackupArena(w, torch.empty(case["n"], dtype=torch.bfloat16, pin_memory=True))
        sub = copes.subspace_build(copes.Layout([case["n"]]), copes.PART_CONTIGUOUS, case["K"], case["k"],
                                   tile_size=case["tile"])
        lo = (case["n"] * case["k"] // case["K"]) & ~3
        buf = torch.empty(max(case["n"] * (case["k"] + 1) // case["K"] - lo, 8), dtype=torch.bfloat16, device="cuda")
        return {"case": case, "arena": arena, "sub": sub, "cfg": _config(case), "partner": es.Partner(buf, lo),
                "rewards": torch.from_numpy(_rewards(case["N"], seed)).cuda()}
    layout = copes.Layout(_numel(case))
    arena = _arena(layout.d_pad, seed, case.get("dtype", "bf16"), case["copies"])
    state = {"case": case, "arena": arena, "layout": layout, "cfg": _config(case), "d": sum(_numel(case)),
             "rewards": torch.from_numpy(_rewards(case["N"], seed)).cuda(), "partner": _partner(arena, case["copies"])}
    if kind == "sync":
        state["step"] = 0
        state["parts"] = es.ChunkPrefetcher(layout, case["K"], lambda s: PARTITION_SEED + s, chunk=case["chunk"])
        state["parts"].prefetch(0)
        return state
    mode, K, k = case["mode"], case["K"], case["k"]
    if mode == "contiguous":
        sub = copes.subspace_build(layout, copes.PART_CONTIGUOUS, K, k, tile_size=case["tile"])
    elif mode == "groups":
        sub = copes.subspace_build(layout, copes.PART_TENSOR_GROUPS, K, k, tile_size=case["tile"],
                                   group_of=workloads.workload(case["layout"]).group_of)
    elif mode in ("hash-lists", "hash-gathered"):
        sub = copes.hash_partition(layout, K, PARTITION_SEED)[k]
    else:
        sub = copes.hash_replay_partition(layout, K, PARTITION_SEED)[k]
        if mode == "hash-mask":
            state["mask"] = torch.empty(int(sub.replay.n_replay_tiles) * 512, dtype=torch.int32, device="cuda")
    state["sub"] = sub
    return state


def _prepare_partition(case, seed):
    """A program that owns its memory: the scratch, and one buffer the K lists are cut from."""
    layout = copes.Layout(_numel(case))
    nbytes = copes.load().copes_hash_workspace_bytes(ctypes.byref(layout.desc), case["K"])
    return {"case": case, "layout": layout, "seed": PARTITION_SEED + seed,
            "scratch": torch.empty(nbytes, dtype=torch.uint8, device="cuda"),
            "lists": torch.zeros(sum(_numel(case)) + case["K"], dtype=torch.int64, device="cuda"),
            "counts": np.zeros(case["K"], np.uint64)}


# ---------------------------------------------------------------------------------- run
def run(state):
    case, kind = state["case"], state["case"]["kind"]
    if kind == "partition":
        return _run_partition(state, case["K"])
    arena = state["arena"]
    if kind == "call":
        return _run_call(state, case, arena)
    if kind == "backup":
        f = es.backup_visit(arena, state["sub"], case["k"], ITERATION, state["cfg"], case["n"], state["rewards"],
                            partner=state["partner"])
        return {"w": arena.w, "backup": arena.backup, "fitness": f}
    if kind == "sync":
        step = state["step"]
        state["step"] = step + 1
        subs = state["parts"].take(step)
        state["parts"].prefetch(step + 1)
        f = es.sync_step(arena, subs, step, state["cfg"], state["d"], state["rewards"], partner=state["partner"])
        return {"master": arena.master, "w": arena.copies, "fitness": f}
    sub = state["sub"]
    if case["mode"] == "hash-gathered":
        copes.gather_master(arena, sub)
    elif case["mode"] == "hash-mask":
        copes.hash_replay_mask(arena, sub, state["mask"])
    f = es.round_robin_visit(arena, sub, case["k"], ITERATION, state["cfg"], state["d"], state["rewards"],
                             partner=state["partner"])
    if case["mode"] == "hash-gathered":
        copes.scatter_master(arena, sub)
    return {"master": arena.master, "w": arena.copies, "fitness": f}


def _run_partition(state, K):
    lib, scratch, lists, counts = copes.load(), state["scratch"], state["lists"], state["counts"]
    layout, stream = ctypes.byref(state["layout"].desc), torch.cuda.current_stream().cuda_stream
    rc = lib.copes_hash_count(layout, K, state["seed"], scratch.data_ptr(), scratch.numel(),
                              counts.ctypes.data_as(ctypes.c_void_p), stream)
    begin = np.concatenate([[0], np.cumsum((counts.astype(np.int64) + 1) // 2 * 2)])  # lists start 16-byte aligned
    ptrs = (ctypes.c_void_p * K)(*[lists.data_ptr() + 8 * int(b) for b in begin[:-1]])
    rc = rc or lib.copes_hash_fill(layout, K, state["seed"], scratch.data_ptr(), scratch.numel(), ptrs, stream)
    if rc:
        raise RuntimeError(copes.last_error())
    return {"lists": lists, "counts": counts.astype(np.int64)}


def _run_call(state, case, arena):
    op, sub, seeds = case["op"], state["sub"], state["seeds"]
    if op == "perturb":
        copes.perturb(arena, sub, int(seeds[0]), SIGMA)
        return arena.w
    if op == "pair":
        copes.perturb_pair(arena, sub, int(seeds[0]), SIGMA, arena.w2)
        return arena.copies
    if op == "two_pairs":
        copes.perturb_two_pairs(arena, sub, int(seeds[0]), int(seeds[1]), SIGMA)
        return arena.copies
    if op == "init":
        copes.init_normal(arena, sub, int(seeds[0]), 0.0, 0.02)
        return [arena.master, arena.w]
    P = case["N"] // 2
    copes.update(arena, sub, state["nid"], state["sign"], state["fitness"], seeds[:P],
                 copes.step_coef(ALPHA, case["N"], SIGMA, copes.COEF_OPENAI))
    return [arena.master, arena.w]


# --------------------------------------------------------------------------------- work
_OPS_NORMAL = 27  # lane-operations of one normal: Philox4x32-10 / 4, uniform, transform


def work(case):
    """bytes: every member's weights written, theta and the context read and written once;
    flops: lane-operations of the normals a pass cannot do without (an antithetic pair
    shares one noise vector) and of the update's sums."""
    d, kind = _d_k(case), case["kind"]
    s = 4 if case.get("dtype") == "fp32" else 2
    if kind == "partition":
        return {"bytes": 8 * d, "flops": 20 * d}
    if kind == "call":
        writes = {"perturb": s, "pair": 2 * s, "two_pairs": 4 * s, "init": 4 + s, "update": 4 + s}[case["op"]]
        reads = 0 if case["op"] == "init" else 4
        normals = {"two_pairs": 2, "update": case["N"] // 2}.get(case["op"], 1)
        return {"bytes": d * (reads + writes), "flops": d * normals * (_OPS_NORMAL + 1)}
    N = case["N"] // case["K"] if kind == "sync" else case["N"]
    P = N if case.get("pairing") == "one_sided" else N // 2
    if kind == "backup":
        return {"bytes": d * (2 * N + 2 + 2 + 2 + 2), "flops": d * P * (2 * _OPS_NORMAL + 1)}
    copies = case["copies"]
    return {"bytes": d * (s * N + 4 + 4 + s * copies), "flops": d * P * (2 * _OPS_NORMAL + 1)}


def tolerance(case):
    """Perturbed and committed bf16 weights may differ by one rounding (2^-7 of a value at
    most) in a few elements of 10^5, which is about 1e-5 in the 2-norm; fp32 masters and
    weights by a few rounding errors (1.5e-7 from 64 bits)."""
    if case["kind"] == "partition":
        return "exact"
    if case["kind"] != "sync" and case.get("dtype") == "fp32":
        return {"rel": 1e-6, "max": 1e-5}
    return {"rel": 5e-5, "max": 1e-2}


# -------------------------------------------------------------------------------- exact
_M0, _M1, _W0, _W1, _MASK = 0xD2511F53, 0xCD9E8D57, 0x9E3779B9, 0xBB67AE85, 0xFFFFFFFF


def _philox(c0, c1, c2, c3, k0, k1):
    """Philox4x32-10 on int64 tensors (or Python ints) holding 32-bit words."""
    for _ in range(10):
        p0, p1 = c0 * _M0, c2 * _M1  # int64 wraps modulo 2^64: the words below are exact
        c0, c1, c2, c3 = ((p1 >> 32) & _MASK) ^ c1 ^ k0, p1 & _MASK, ((p0 >> 32) & _MASK) ^ c3 ^ k1, p0 & _MASK
        k0, k1 = (k0 + _W0) & _MASK, (k1 + _W1) & _MASK
    return c0, c1, c2, c3


def _lattice():
    """Phi^-1 at the 2^22 uniforms ((2 i + 1) 2^-23)."""
    u = (2 * torch.arange(1 << 22, device="cuda", dtype=torch.float64) + 1) * 2.0**-23
    return torch.special.ndtri(u)


def _normal(word, lattice):
    return lattice[(word & 0x7FFFFE) >> 1]


def _member_seeds(iteration, k, P):
    return [x[0] | (x[1] << 32) for x in (_philox(j, k, iteration, 3, BASE_SEED, 0) for j in range(P))]


def _noise_blocks(seeds, q0, q1, tag, lattice):
    """Normals of the counters [q0, q1) for each seed, [4 (q1 - q0)] each."""
    q = torch.arange(q0, q1, device="cuda", dtype=torch.int64)
    for s in seeds:
        x = _philox(q & _MASK, q >> 32, torch.zeros_like(q), tag, s & _MASK, s >> 32)
        yield _normal(torch.stack(x, 1).reshape(-1), lattice)


def _add_noise(out, ranges, seeds, weights, tag=0):
    """out[g] += sum_j weights[j] eps_j[g] over the ranges."""
    lattice, step = _lattice(), 1 << 22
    for b, e in ranges:
        for lo in range(b & ~3, e, 4 * step):
            hi = min(lo + 4 * step, (e + 3) & ~3)
            i, j = max(lo, b), min(hi, e)
            acc = torch.zeros(j - i, device="cuda", dtype=torch.float64)
            for w, eps in zip(weights, _noise_blocks(seeds, lo // 4, hi // 4, tag, lattice)):
                acc.add_(eps[i - lo:j - lo], alpha=w)
            out[i:j] += acc


def _shape(rewards, mode):
    r = rewards.astype(np.float64)
    if mode == "none":
        return r
    if mode == "zscore":
        return np.zeros_like(r) if np.all(r == r[0]) else (r - r.mean()) / r.std()
    if r.size == 1:
        return np.zeros(1)
    rank = (r[:, None] > r[None]).sum(1) + 0.5 * ((r[:, None] == r[None]).sum(1) - 1)
    return rank / (r.size - 1) - 0.5


def _weights(f, pairing, coef):
    """coef * w_j: the members of noise vector j folded."""
    return [float(coef * x) for x in (f if pairing == "one_sided" else f[0::2] - f[1::2])]


def _hash_members(case):
    """Global indices of subspace k of the hash partition."""
    numel, out, off = _numel(case), [], 0
    for t, n in enumerate(numel):
        for lo in range(0, n, 1 << 24):
            hi = min(lo + (1 << 24), n)
            q = torch.arange(lo // 4, (hi + 3) // 4, device="cuda", dtype=torch.int64)
            x = _philox(q & _MASK, q >> 32, torch.full_like(q, t), 2, PARTITION_SEED & _MASK, 0)
            bucket = (torch.stack(x, 1).reshape(-1)[:hi - lo] * case["K"]) >> 32
            out.append(torch.nonzero(bucket == case["k"]).reshape(-1) + (off + lo))
        off = (off + n + 63) // 64 * 64
    return torch.cat(out)


def _add_noise_at(out, index, seeds, weights):
    lattice = _lattice()
    for lo in range(0, index.numel(), 1 << 22):
        g = index[lo:lo + (1 << 22)]
        acc = torch.zeros(g.numel(), device="cuda", dtype=torch.float64)
        for s, w in zip(seeds, weights):
            x = torch.stack(_philox((g >> 2) & _MASK, g >> 34, torch.zeros_like(g), 0, s & _MASK, s >> 32), 1)
            acc.add_(_normal(x.gather(1, (g & 3)[:, None]).reshape(-1), lattice), alpha=w)
        out[g] += acc


def _add_noise_chunks(out, case, f):
    """Algorithm 1's composed update: every chunk's elements take its subspace's noise."""
    K, C, n = case["K"], case["chunk"], sum(_numel(case))
    n_k = case["N"] // K
    n_chunks = (out.numel() + C - 1) // C
    c = torch.arange(n_chunks, device="cuda", dtype=torch.int64)
    key = _philox(c, torch.zeros_like(c), torch.zeros_like(c), 4, PARTITION_SEED & _MASK, 0)[0]
    rank = torch.empty_like(c)
    rank[torch.argsort((key << 20) | c)] = c
    owner = rank * K // n_chunks
    seeds = torch.tensor([_wrap(_member_seeds(0, k, n_k // 2)) for k in range(K)], device="cuda")  # [K, P]
    w = torch.tensor([_weights(f[k * n_k:(k + 1) * n_k], "antithetic", ALPHA / n_k) for k in range(K)],
                     device="cuda", dtype=torch.float64)
    lattice, per = _lattice(), max(1, (1 << 24) // C)
    for lo in range(0, n_chunks, per):
        own = owner[lo:lo + per]
        q = (torch.arange(own.numel() * C // 4, device="cuda", dtype=torch.int64) + lo * C // 4).reshape(-1, C // 4)
        acc = torch.zeros(own.numel(), C, device="cuda", dtype=torch.float64)
        for j in range(n_k // 2):
            s = seeds[own, j][:, None]
            x = _philox(q & _MASK, q >> 32, torch.zeros_like(q), 0, s & _MASK, (s >> 32) & _MASK)
            acc += w[own, j][:, None] * _normal(torch.stack(x, 2).reshape(-1, C), lattice)
        i, j = lo * C, min((lo + own.numel()) * C, n)
        out[i:j] += acc.reshape(-1)[:j - i]


def _wrap(seeds):
    return [s - (1 << 64) if s >> 63 else s for s in seeds]


def exact(case, seed):
    kind = case["kind"]
    if kind == "partition":
        return None  # whole numbers
    if kind == "call":
        return _exact_call(case, seed)
    f = _shape(_rewards(case["N"], seed), case.get("shaping", "zscore"))
    fit = torch.from_numpy(f)
    if kind == "backup":
        t = _theta(case["n"], seed).to(torch.bfloat16).double()
        b, e = case["n"] * case["k"] // case["K"], case["n"] * (case["k"] + 1) // case["K"]
        w = _weights(f, "antithetic", ALPHA / (case["N"] * SIGMA))
        _add_noise(t, [(b, e)], _member_seeds(ITERATION, case["k"], len(w)), w)
        return {"w": t, "backup": None, "fitness": fit}
    d_pad = workloads.layout_offsets([workloads.Tensor("", m, "") for m in _numel(case)])[-1]
    t = _theta(d_pad, seed).double()
    if kind == "sync":
        _add_noise_chunks(t, case, f)
    else:
        w = _weights(f, case["pairing"], ALPHA / (case["N"] * case["sigma"]))
        seeds = _member_seeds(ITERATION, case["k"], len(w))
        if case["mode"].startswith("hash"):
            _add_noise_at(t, _hash_members(case), seeds, w)
        else:
            _add_noise(t, _span(case), seeds, w)
    return {"master": t, "w": [t] * case["copies"], "fitness": fit}


def _exact_call(case, seed):
    op, r = case["op"], [(case["begin"], case["end"])]
    P = case["N"] // 2
    seeds = _member_seeds(ITERATION, 0, max(P, 2))
    theta = _theta(case["n"], seed).double()

    def moved(s, sigma):
        out = theta.clone()
        _add_noise(out, r, [s], [sigma])
        return out

    if op == "perturb":
        return moved(seeds[0], SIGMA)
    if op == "pair":
        return [moved(seeds[0], SIGMA), moved(seeds[0], -SIGMA)]
    if op == "two_pairs":
        return [moved(s, x) for s in seeds[:2] for x in (SIGMA, -SIGMA)]
    if op == "init":
        out = theta.clone()
        out[case["begin"]:case["end"]] = 0
        _add_noise(out, r, [seeds[0]], [0.02], tag=1)
        return [out, out]
    _add_noise(theta, r, seeds[:P], _weights(_fitness(case["N"], seed).astype(np.float64), "antithetic",
                                             ALPHA / (case["N"] * SIGMA)))
    return [theta, theta]
