"""Performance cases: what a user of the library has it do, through the binding's public calls.

A deployment is a client that encrypts queries and decrypts scores, and a stateless server that keeps contexts, evaluation
keys and workspaces and scores one encrypted query after another against levels of candidate rows.  The listed cases cover
that round trip: levels whose rows arrive per query (device-resident, or from page-locked host memory), levels whose encoded
candidates stay resident (one query, or a batch of queries), an encrypted database, the projection of a query under
encryption, the membership circuit, and the client's half.  `draw` gives further cases of the same ranges.

A context with its keys belongs to one client and serves all of its queries, so states of the same parameters share one;
queries, candidate rows, their encodings and all output buffers belong to a state.
"""
import functools
import math

import numpy as np
import torch

from paper_2608_21131_b200 import binding, synth

KEY_SEED = 1
DEVICE = "cuda:0"
LAZY, HORNER = "lazy", "horner"  # order of evaluation of the giant steps (Horner is the library's default)


# ------------------------------------------------------------------------------------------------------------ the cases


def listed():
    return [
        # the smallest level: 4,096 rows of dimension 64 on the small ring with 30-bit primes; a chain of short launches
        dict(name="toy_level", kind="level", primes="toy", logN=12, L=2, R=64, B=8, dim=64, rows=4096, giant=HORNER),
        # coarse level of the billion-row hierarchy: 1,000 centroids of dimension 96 in one mostly empty block
        dict(name="coarse_1000", kind="level", primes="q50", logN=16, L=4, R=128, B=32, dim=96, rows=1000, giant=LAZY),
        # rerank level of the 512-dimensional hierarchy: about 100k fetched rows, last block ragged, default giant-step order
        dict(name="rerank_97976", kind="level", primes="q50", logN=16, L=4, R=128, B=32, dim=128, rows=97976, giant=HORNER),
        # the face-like flat level: every row scored for one query, rows resident on the device
        dict(name="face_222049", kind="level", primes="q50", logN=16, L=4, R=128, B=32, dim=128, rows=222049, giant=LAZY),
        # the same from page-locked host buffers: query and rows go up, score ciphertexts come home
        dict(name="face_host_222049", kind="host", primes="q50", logN=16, L=4, R=128, B=32, dim=128, rows=222049, giant=LAZY),
        # top of the padding sweep: 2^18 wanted rows inflated four times, on the smaller ring (64 blocks)
        dict(name="sweep_1048576", kind="level", primes="q50", logN=15, L=4, R=128, B=32, dim=128, rows=1048576, giant=LAZY),
        # warm level: the encoded candidates of a hot region stay resident, every query brings only itself
        dict(name="resident_1000000", kind="resident", primes="q50", logN=16, L=4, R=128, B=32, dim=128, rows=1000000, queries=1, giant=LAZY),
        # cross-query batching: several clients' queries (here of one client) against one resident coarse level
        dict(name="batch8_65536", kind="resident", primes="q50", logN=16, L=4, R=128, B=32, dim=128, rows=65536, queries=8, giant=HORNER),
        # encrypted database: candidate diagonals are ciphertexts, resident; one relinearisation per giant step
        dict(name="encrypted_65536", kind="ctdb", primes="q50", logN=15, L=4, R=128, B=32, dim=128, rows=65536, giant=HORNER),
        # rank reduction 512 -> 128 of one encrypted query, matrix packed by windows
        dict(name="project_512", kind="project", primes="q50", logN=16, L=4, R=128, B=8, dim=512, rows=0, giant=LAZY),
        # threshold decision for every row of the face-like level under encryption: depth 11 on 12 primes
        dict(name="membership_222049", kind="membership", primes="chain", logN=15, L=12, R=128, B=32, dim=128, rows=222049, giant=HORNER),
        # the client's half of a round trip: encrypt the next query, decrypt the last level's score ciphertexts
        dict(name="client_222049", kind="client", primes="q50", logN=16, L=4, R=128, B=32, dim=128, rows=222049, giant=LAZY),
    ]


def draw(rng):
    kind = rng.choice(["level"] * 5 + ["host", "host", "resident", "resident", "batch", "ctdb", "project", "membership", "client"])

    def rows(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    giant = rng.choice([LAZY, HORNER])
    if kind == "membership":
        return dict(kind=kind, primes="chain", logN=15, L=12, R=128, B=32, dim=128, rows=rows(300, 222049), giant=HORNER)
    if kind == "project":
        return dict(kind=kind, primes="q50", logN=rng.choice([15, 16]), L=4, R=rng.choice([64, 128]), B=rng.choice([8, 16]),
                    dim=rng.choice([256, 512]), rows=0, giant=giant)
    if kind == "level" and rng.random() < 0.2:
        return dict(kind=kind, primes="toy", logN=12, L=2, R=64, B=8, dim=rng.randint(17, 64), rows=rows(1, 60000), giant=giant)
    logN = rng.choice([14, 15, 15, 16, 16, 16])
    R = rng.choice([64, 128, 128])
    case = dict(kind=kind, primes="q50", logN=logN, L=rng.choice([2, 3, 4, 4]), R=R, B=rng.choice([16, 32]),
                dim=rng.choice([R, R, rng.randint(R // 2, R)]), rows=0, giant=giant)
    if kind in ("level", "host"):
        case["rows"] = rows(1, 700000)
    elif kind == "client":
        case["rows"] = rows(1, 222049)
    elif kind == "ctdb":
        case["logN"] = min(logN, 15)
        case["rows"] = rows(1, 65536)
        case["giant"] = HORNER
    else:
        case["kind"] = "resident"
        case["queries"] = rng.randint(2, 8) if kind == "batch" else 1
        case["rows"] = rows(1, 65536 if kind == "batch" else 1000000)
    return case


# ----------------------------------------------------------------------------------------- contexts and keys of a client


def _is_prime(n):
    if any(n % b == 0 for b in (2, 3, 5, 7, 11, 13, 17, 19, 23, 29, 31, 37)):
        return False
    d, r = n - 1, 0
    while d % 2 == 0:
        d, r = d // 2, r + 1
    for b in (2, 3, 5, 7, 11, 13, 17, 19, 23, 29, 31, 37):  # deterministic far beyond 64 bits
        x = pow(b, d, n)
        if x in (1, n - 1):
            continue
        for _ in range(r - 1):
            x = x * x % n
            if x == n - 1:
                break
        else:
            return False
    return True


def _primes_below(bits, count, logN):
    out, c = [], (1 << bits) - (2 << logN) + 1
    while len(out) < count:
        if _is_prime(c):
            out.append(c)
        c -= 2 << logN
    return out


# the membership circuit: degree-7 square root, three sign iterations, 45-bit scale
MEM = dict(deg=7, iters=3, log_scale=45, tau=0.45, t_lo=0.05, t_hi=1.0, kappa=0.5)


@functools.lru_cache(maxsize=None)
def _membership_chain(logN):
    """primes in the order of the chain (the first one large, the others consumed from the end) and the special prime"""
    n_thr = 5
    p45 = _primes_below(MEM["log_scale"], n_thr + MEM["iters"], logN)
    p46 = _primes_below(MEM["log_scale"] + 1, MEM["iters"], logN)
    consumed = p45[:n_thr]
    for i in range(MEM["iters"]):
        consumed += [p45[n_thr + i], p46[i]]
    return tuple(_primes_below(58, 1, logN) + consumed[::-1]), _primes_below(60, 1, logN)[0]


def _params(case):
    if case["primes"] == "toy":
        return synth.ParamSet("case", case["logN"], synth.Q30, synth.P31, 25, case["R"], case["B"], -10)
    if case["primes"] == "chain":
        q, p = _membership_chain(case["logN"])
        return synth.ParamSet("case", case["logN"], q, p, MEM["log_scale"], case["R"], case["B"], -10)
    return synth.ParamSet("case", case["logN"], synth.Q50[: case["L"]], synth.P60, 40, case["R"], case["B"], -18)


def _uniform(rng, q, lead, N):
    """uint64 [*lead][len(q)][N], entry uniform in [0, q_i)"""
    out = np.empty(tuple(lead) + (len(q), N), dtype=np.uint64)
    for i, qi in enumerate(q):
        out[..., i, :] = rng.integers(0, qi, size=tuple(lead) + (N,), dtype=np.uint64)
    return out


def _errors(rng, shape):
    return np.rint(3.2 * rng.standard_normal(shape)).astype(np.int8)


@functools.lru_cache(maxsize=None)
def _server(ps, giant, relin):
    """(context, secret key): the context with the rotation keys of its scoring path loaded"""
    ctx = binding.Context(ps)
    rots = list(range(1, ps.B + 1)) + ([g * ps.B for g in range(2, ps.G)] if giant == LAZY else [])
    s, evk = ctx.keygen_seeded(KEY_SEED, rots)
    ctx.load_keys(evk, rots)
    if giant == LAZY:
        ctx.set_tuning(binding.TUNE_GIANT_LAZY, 1)
    if relin:
        rng = np.random.default_rng(KEY_SEED)
        a, e = _uniform(rng, ps.q + (ps.p,), (ps.L,), ps.N), _errors(rng, (ps.L, ps.N))
        ctx.load_keys(ctx.keygen_relin_from_samples(s, a, e)[None], [0])
    return ctx, s


@functools.lru_cache(maxsize=None)
def _projector(ps, dim, giant):
    """(top context, middle context, query-encryption context, secret key) of the packed projection dim -> R"""
    top, mid = binding.Context(ps), binding.Context(ps.with_(q=ps.q[:-1]))
    rots_top = list(range(1, ps.B)) + [top.n - ps.R + b for b in range(1, ps.B)]
    rots_mid = sorted({g * ps.B for g in range(1, ps.G)} | {ps.R << t for t in range((dim // ps.R).bit_length() - 1)})
    rots = sorted(set(rots_top) | set(rots_mid))
    s, evk = top.keygen_seeded(KEY_SEED, rots)
    top.load_keys(evk[[rots.index(r) for r in rots_top]], rots_top)
    mid.load_keys(binding.restrict_keys(evk[[rots.index(r) for r in rots_mid]], ps.L, ps.L - 1), rots_mid)
    mid.set_tuning(binding.TUNE_GIANT_LAZY, 1 if giant == LAZY else 0)
    return top, mid, binding.Context(ps.with_(R=dim, B=1)), s


@functools.lru_cache(maxsize=None)
def _membership(ps):
    """(contexts by level, scorer, query-encryption context, secret key) of the membership circuit"""
    levels = np.zeros(2, dtype=np.int32)
    binding.load_library().hann_membership_levels(MEM["deg"], MEM["iters"], levels[0:].ctypes.data, levels[1:].ctypes.data)
    L, score_level = int(levels[0]), int(levels[1])
    arith = [binding.Context(ps.with_(q=ps.q[:l], R=1, B=1)) for l in range(1, L + 1)]
    scorer, qctx = binding.Context(ps.with_(q=ps.q[:score_level])), binding.Context(ps.with_(B=1))
    s = None
    fold = [1 << t for t in range(ps.R.bit_length() - 1)]
    for r in sorted(set(range(1, ps.B + 1)) | set(fold)):  # one rotation at a time: a key of the full chain is large
        s, evk = arith[L - 1].keygen_seeded(KEY_SEED, [r])
        if r in fold:
            arith[L - 2].load_keys(binding.restrict_keys(evk, L, L - 1), [r])
        if r <= ps.B:
            scorer.load_keys(binding.restrict_keys(evk, L, score_level), [r])
    rng = np.random.default_rng(KEY_SEED)
    rlk = arith[L - 1].keygen_relin_from_samples(s, _uniform(rng, ps.q + (ps.p,), (L,), ps.N), _errors(rng, (L, ps.N)))
    for l in range(2, L + 1):
        arith[l - 1].load_keys(binding.restrict_keys(rlk, L, l)[None], [0])
    return arith, scorer, qctx, s


# ------------------------------------------------------------------------------------------------------------- inputs


def _rows(seed, n, dim):
    """n unit-norm rows of a clustered corpus (256 unit-norm means, noise of norm about 0.6 before normalisation)"""
    gen = torch.Generator(device=DEVICE).manual_seed(seed)
    mu = torch.nn.functional.normalize(torch.randn(256, dim, generator=gen, device=DEVICE), dim=1)
    x = mu[torch.randint(256, (n,), generator=gen, device=DEVICE)]
    x += torch.randn(n, dim, generator=gen, device=DEVICE) * (0.6 / math.sqrt(dim))
    return torch.nn.functional.normalize(x, dim=1).contiguous()


def _query_near(rng, row):
    q = row.astype(np.float64) + rng.standard_normal(row.shape[0]) * (0.1 / math.sqrt(row.shape[0]))
    return (q / np.linalg.norm(q)).astype(np.float32)


def _encrypted(ctx, ps, s, q, rng):
    return ctx.encrypt_query(s, q, _uniform(rng, ps.q, (), ps.N), _errors(rng, (ps.N,)))


def prepare(case, seed):
    rng = np.random.default_rng(seed)
    ps = _params(case)
    kind = case["kind"]
    st = dict(kind=kind, case=case)
    if kind == "project":
        return _prepare_project(st, case, ps, rng)
    if kind == "membership":
        return _prepare_membership(st, case, ps, rng, seed)
    ctx, s = _server(ps, case["giant"], kind == "ctdb")
    n_rows, dim = case["rows"], case["dim"]
    rows = _rows(seed, n_rows, dim)
    nb, nq = ctx.n_blocks(n_rows), case.get("queries", 1)
    near = [rows[(i + 1) * n_rows // (nq + 2)].cpu().numpy() for i in range(nq)]
    cts = [_encrypted(ctx, ps, s, _query_near(rng, x), rng) for x in near]
    st.update(ctx=ctx, nb=nb)
    if kind == "host":
        st["ct"] = torch.from_numpy(cts[0].view(np.int64)).pin_memory()
        st["rows"] = rows.cpu().pin_memory()
        st["ws"] = ctx.alloc(ctx.level_host_bytes(n_rows))
        st["out"] = torch.empty((nb, 2, ctx.L, ctx.N), dtype=torch.int64).pin_memory()
        return st
    ct_dev = [ctx.import_(binding.KIND_CT, ct, 1) for ct in cts]
    ws = ctx.workspace(min(nb * nq, 64))
    baby = ctx.alloc(nq * ctx.sizeof(binding.SIZE_BABY))
    inner = ctx.alloc(nq * nb * ctx.sizeof(binding.SIZE_INNER))
    score = ctx.alloc(nq * nb * ctx.sizeof(binding.SIZE_CT))
    st.update(ct=ct_dev, ws=ws, baby=baby, inner=inner, score=score, nq=nq)
    if kind in ("level", "client"):
        st.update(rows=rows, pt=ctx.alloc(nb * ctx.sizeof(binding.SIZE_PT_BLOCK)))
    if kind == "client":
        # the last level's scores as they came home, and what the client draws for its next query
        ctx.query_level(ct_dev[0], rows, ws, baby, st["pt"], inner, score)
        home = ctx.export(binding.KIND_CT, score, nb)
        return dict(kind=kind, case=case, ctx=ctx, s=s, home=home, q=_query_near(rng, near[0]), a=_uniform(rng, ps.q, (), ps.N), e=_errors(rng, (ps.N,)))
    if kind == "resident":
        st["pt"] = ctx.encode_candidates(rows, ws)
    if kind == "ctdb":
        pt = ctx.encode_candidates(rows, ws)
        ptw, dbw = ctx.sizeof(binding.SIZE_PT_BLOCK) // 8, ctx.sizeof(binding.SIZE_CTDB_BLOCK) // 8
        st["db"] = ctx.alloc(nb * dbw * 8)
        for blk in range(nb):
            ctx.encrypt_block(s, pt[blk * ptw:(blk + 1) * ptw], _uniform(rng, ps.q, (ps.R,), ps.N), _errors(rng, (ps.R, ps.N)),
                              st["db"][blk * dbw:(blk + 1) * dbw])
    return st


def _prepare_project(st, case, ps, rng):
    top, mid, qctx, s = _projector(ps, case["dim"], case["giant"])
    W = np.linalg.qr(rng.standard_normal((case["dim"], ps.R)))[0].astype(np.float32)
    q = rng.standard_normal(case["dim"])
    ct = _encrypted(qctx, ps, s, (q / np.linalg.norm(q)).astype(np.float32), rng)
    lo, hi = top.project_masks(50, top.workspace(1))
    wpt = mid.project_enrol(torch.from_numpy(W).to(DEVICE), 50, mid.workspace(1))
    st.update(top=top, mid=mid, ct=top.import_(binding.KIND_CT, ct, 1), lo=lo, hi=hi, wpt=wpt,
              ws=top.alloc(top.lib.hann_project_bytes(top.h, mid.h)))
    return st


def _prepare_membership(st, case, ps, rng, seed):
    arith, scorer, qctx, s = _membership(ps)
    top = arith[-1]
    lam = math.sqrt(2.0 / (MEM["t_hi"] - MEM["t_lo"]) * ps.q[-1] / 2.0 ** MEM["log_scale"])
    k = np.arange(MEM["deg"] + 1)
    nodes = np.cos(np.pi * (k + 0.5) / (MEM["deg"] + 1))
    vals = MEM["kappa"] * MEM["tau"] * np.sqrt(0.5 * (MEM["t_hi"] - MEM["t_lo"]) * nodes + 0.5 * (MEM["t_hi"] + MEM["t_lo"]))
    coef = np.array([2.0 / (MEM["deg"] + 1) * np.sum(vals * np.cos(np.pi * j * (k + 0.5) / (MEM["deg"] + 1))) for j in k])
    coef[0] *= 0.5
    rows = _rows(seed, case["rows"], case["dim"])
    q = 0.7 * _query_near(rng, rows[case["rows"] // 3].cpu().numpy())
    ct = _encrypted(qctx, ps, s, (lam * q.astype(np.float64)).astype(np.float32), rng)
    nb = scorer.n_blocks(case["rows"])
    pt = scorer.encode_candidates((rows * (MEM["kappa"] / lam)).contiguous(), scorer.workspace(nb))
    st.update(arith=arith, scorer=scorer, R=ps.R, coef=coef, ct=top.import_(binding.KIND_CT, ct, 1), pt=pt, nb=nb)
    return st


# --------------------------------------------------------------------------------------------------------------- a pass


def run(st):
    kind = st["kind"]
    if kind == "level":
        return st["ctx"].query_level(st["ct"][0], st["rows"], st["ws"], st["baby"], st["pt"], st["inner"], st["score"])
    if kind == "host":
        return st["ctx"].score_level_host(st["ct"], st["rows"], st["ws"], st["out"])
    if kind in ("resident", "ctdb"):
        ctx, ws, nb, nq = st["ctx"], st["ws"], st["nb"], st["nq"]
        per = st["baby"].numel() // nq
        for i, ct in enumerate(st["ct"]):
            ctx.query_prepare(ct, ws, st["baby"][i * per:(i + 1) * per])
        if kind == "ctdb":
            ctx.score_level_ctdb(st["baby"], st["db"], nb, ws, st["inner"])
        elif nq == 1:
            ctx.score_level(st["baby"], st["pt"], nb, ws, st["inner"])
        else:
            ctx.score_level_batch(st["baby"], nq, st["pt"], nb, ws, st["inner"])
        return ctx.rotate_sum(st["inner"], nq * nb, ws, st["score"])
    if kind == "project":
        return st["top"].project_query(st["mid"], st["ct"], st["lo"], st["hi"], st["wpt"], st["case"]["dim"], st["ws"])
    if kind == "membership":
        out, scale = binding.membership_decide(st["arith"], st["scorer"], st["R"], MEM["deg"], MEM["iters"], MEM["log_scale"], MEM["tau"],
                                               MEM["t_lo"], MEM["t_hi"], st["coef"], st["ct"], st["pt"], st["nb"])
        return {"decision": out, "scale": scale}
    ctx = st["ctx"]
    ct = ctx.encrypt_query(st["s"], st["q"], st["a"], st["e"])
    return {"query": ct.view(np.int64), "scores": ctx.decrypt_scores(st["s"], st["home"])}


# ------------------------------------------------------------------------------------------------- work and tolerance


def work(case):
    """Bytes: inputs, keys and resident data read once, results written once.  Operations: binary64 operations of the
    method's transforms (8 per modular butterfly, 10 per FFT butterfly) and products (4 per product and sum)."""
    logN, L, R, B, dim, rows = (case[k] for k in ("logN", "L", "R", "B", "dim", "rows"))
    N, n, G = 1 << logN, 1 << (logN - 1), R // B
    W = 8 * N
    ct, key = 2 * L * W, 2 * L * (L + 1) * W
    nb, nq = -(-rows // n), case.get("queries", 1)
    T = N // 2 * logN * 8  # one transform

    def keyswitch(l, items=1):  # digits, lifts, key product, ModDown
        return items * ((l + 2 + l * (l + 1) + 2 * l) * T + l * 2 * (l + 1) * N * 4)

    def hoisted(l, count):
        return (l + l * (l + 1)) * T + count * ((2 + 2 * l) * T + l * 2 * (l + 1) * N * 4)

    encode = R * (n // 2 * (logN - 1) * 10 // 2 + L * T // 2)  # a real FFT, half of every limb's transform
    if case["giant"] == LAZY:
        giant_keys, giant = G - 1, lambda l: (G - 1) * ((l + l * (l + 1)) * T + l * 2 * (l + 1) * N * 4) + (2 + 2 * l) * T
    else:
        giant_keys, giant = min(1, G - 1), lambda l: keyswitch(l, G - 1)
    kind = case["kind"]
    if kind == "client":
        per = (2 * L + L) * T + n // 2 * (logN - 1) * 10  # two transforms forward, one back, a complex FFT, per ciphertext
        return {"bytes": ct + nb * (ct + n * 8), "flops": nb * per + 3 * L * T}
    if kind == "project":
        folds = (dim // R).bit_length() - 1
        mid_key = 2 * (L - 1) * L * W
        flops = 2 * hoisted(L, B - 1) + 4 * B * L * N * 4 + (2 * B + 2) * L * T + 2 * R * (L - 1) * N * 4 + giant(L - 1) + keyswitch(L - 1, folds)
        return {"bytes": ct + 2 * (B - 1) * key + 2 * B * L * W // 2 + R * (L - 1) * W // 2 + (giant_keys + folds) * mid_key + 2 * (L - 2) * W,
                "flops": flops}
    if kind == "membership":
        # products at every level with a relinearisation and a rescale each, folds of the norm, the scorer on eight primes
        S, folds = 8, R.bit_length() - 1
        rescale = lambda l: 2 * l * T
        flops = keyswitch(12) + rescale(12) + folds * keyswitch(11) + sum(k * (keyswitch(l) + rescale(l)) for l, k in ((11, 1), (10, 2), (9, 3)))
        flops += hoisted(S, B - 1) + nb * (R * 2 * S * N * 4 + keyswitch(S, G - 1) + rescale(S) + sum(keyswitch(l) + rescale(l) for l in range(7, 1, -1)))
        keyb = lambda l: 2 * l * (l + 1) * W
        bytes_ = ct + nb * R * S * W // 2 + B * keyb(S) + folds * keyb(11) + sum(keyb(l) for l in range(2, 13)) + nb * 2 * W
        return {"bytes": bytes_, "flops": flops}
    flops = nq * hoisted(L, B - 1) + nq * nb * giant(L)
    bytes_ = nq * ct + (B - 1 + giant_keys) * key + nq * nb * ct
    if kind == "ctdb":
        bytes_ += nb * R * ct + key
        flops += nb * (R * 4 * L * N * 4 + keyswitch(L, G))
    else:
        flops += nq * nb * R * 2 * L * N * 4
        if kind == "resident":
            bytes_ += nb * R * L * W // 2
        else:
            bytes_ += rows * dim * 4
            flops += nb * encode
    return {"bytes": bytes_, "flops": flops}


def tolerance(case):
    """Ciphertexts are residues and compare bit for bit.  Decrypted scores are binary64 results of a CRT, a twist and an FFT of n
    points: two evaluations of those with their sums in another order differ by 3.1e-16 to 3.4e-16 (2-norm, n = 2^13 .. 2^15)."""
    return {"rel": 1.4e-15, "differ": 0.0} if case["kind"] == "client" else "exact"
