"""The measured workloads of the share-domain uniqueness check, each through the public binding.

Kinds of case:
  request   a context with a resident database answers requests (submit_queries, fetch_bit_shares,
            ipc_release), `requests` of them submitted together and fetched in order;
  serve     the continuous-batching loop answers a burst of requests of several sizes;
  persons   both eyes and inner-batch matching (ipc_check_persons);
  stage     the stage-level calls for one chunk that the caller owns: query preparation, the six
            ring GEMMs, the comparison and the OR tree, with every message and share returned;
  compare   the comparison phase and the OR tree alone, on given dot-product components;
  enrol     client encoding and sharing of new rows and their split into resident limb planes.

Options: `path` (tc replicated sharing on tcgen05, tcg Galois-ring Shamir shares, i8mix / i8mma / i32
the integer pipes), `plain` (protocol 1, public masks), `lift` (mpc, const, none: the lifting variants),
`rows`, `queries`, `rot` (rotations), `cols` (columns of the 16 x cols x 4 code; 200 is an iris code).
Codes are Bernoulli(0.5) bits, masks about Bernoulli(0.9); some queries are rotated near-duplicates
of a database row (10 % of the bits flipped), as a returning person's would be.
"""
import numpy as np
import torch

import paper_2405_04463_gb300 as ipc

THR_A = 16384           # MATCH_RATIO 0.375: a match is 4 dot > ml
DB_SEED, Q_SEED = 0xDB5EED, 0x0E5EED
M32 = 0xFFFFFFFF


def listed():
    return [
        # the smallest workload: a handful of codes without rotations against a small register
        {"name": "tiny_request", "kind": "request", "path": "tc", "rows": 1000, "queries": 4, "rot": 1, "cols": 200,
         "requests": 1, "lift": "mpc", "plain": False, "host": True},
        # persons arriving one by one at several stations: single-code requests, submitted as they come
        {"name": "single_codes", "kind": "request", "path": "tc", "rows": 100000, "queries": 1, "rot": 31, "cols": 200,
         "requests": 4, "lift": "mpc", "plain": False, "host": True},
        # the benchmark's step: 100,000 rows x 32 codes x 31 rotations, replicated sharing, host shares
        {"name": "headline_100k_x32", "kind": "request", "path": "tc", "rows": 100000, "queries": 32, "rot": 31,
         "cols": 200, "requests": 1, "lift": "mpc", "plain": False, "host": True},
        # the deployed sharing at a serving-sized batch (mean of 1..256 codes)
        {"name": "galois_100k_x128", "kind": "request", "path": "tcg", "rows": 100000, "queries": 128, "rot": 31,
         "cols": 200, "requests": 1, "lift": "mpc", "plain": False, "host": False},
        # protocol 1 (public masks), an odd register and an odd batch
        {"name": "plain_masks_odd", "kind": "request", "path": "tcg", "rows": 70003, "queries": 9, "rot": 31,
         "cols": 200, "requests": 1, "lift": "mpc", "plain": True, "host": False},
        # ConstLift: mask shares and mask dot products over Z_2^32
        {"name": "constlift_30k_x16", "kind": "request", "path": "tc", "rows": 30000, "queries": 16, "rot": 31,
         "cols": 200, "requests": 1, "lift": "const", "plain": False, "host": False},
        # the integer-only path (int8 mma.sync with dp4a)
        {"name": "integer_8k_x8", "kind": "request", "path": "i8mix", "rows": 8192, "queries": 8, "rot": 31,
         "cols": 200, "requests": 1, "lift": "mpc", "plain": False, "host": False},
        # a burst of mixed requests through the serving loop
        {"name": "serve_burst", "kind": "serve", "path": "tc", "rows": 80000, "sizes": "5,48,17,1,25", "rot": 31,
         "cols": 200},
        # both eyes of a batch of persons, with inner-batch matching
        {"name": "persons_2x40k_x8", "kind": "persons", "path": "tcg", "rows": 40000, "queries": 8, "rot": 31,
         "cols": 200},
        # a caller's own pipeline on one ragged chunk, every message kept
        {"name": "stages_ragged", "kind": "stage", "path": "tc", "rows": 9973, "queries": 7, "rot": 31, "cols": 200},
        # the comparison phase of one resident chunk at the benchmark's width
        {"name": "compare_chunk", "kind": "compare", "rows": 65536, "queries": 32, "rot": 31, "mode": "lift"},
        # enrolment of a batch of new rows
        {"name": "enrol_8k", "kind": "enrol", "rows": 8192, "cols": 200, "ring": 16},
    ]


def _log(rng, lo, hi):
    return max(lo, min(hi, int(round(lo * (hi / lo) ** rng.random()))))


def _cost(c):
    """A pass in units of one tcgen05 limb product: the integer pipes run at a small part of that rate."""
    slow = {"i8mix": 6.5, "i8mma": 11, "i32": 15}.get(c.get("path"), 1)
    return work(c)["flops"] * slow


def draw(rng):
    cap = max(_cost(c) for c in listed())
    while True:
        kind = rng.choice(["request"] * 6 + ["serve", "persons", "stage", "compare", "enrol"])
        rot, cols = rng.choice([31, 31, 31, rng.randint(1, 30)]), rng.choice([200, 200, 200, 8 * rng.randint(4, 32)])
        if kind == "request":
            c = {"kind": kind, "path": rng.choice(["tc"] * 4 + ["tcg"] * 3 + ["i8mix", "i8mma", "i32"]),
                 "rows": _log(rng, 300, 100000), "queries": _log(rng, 1, 128), "rot": rot, "cols": cols,
                 "requests": rng.choice([1, 1, 2]), "lift": "mpc", "plain": False, "host": rng.random() < 0.5}
            if c["queries"] * c["requests"] < 4:
                c["requests"] = 4
            if c["path"] == "tc" and rng.random() < 0.35:
                c["lift"] = rng.choice(["const", "none"])
            elif c["path"] in ("tc", "tcg") and rng.random() < 0.25:
                c["plain"] = True
        elif kind == "serve":
            c = {"kind": kind, "path": rng.choice(["tc", "tcg"]), "rows": _log(rng, 2000, 100000),
                 "sizes": ",".join(str(_log(rng, 1, 64)) for _ in range(rng.randint(3, 6))), "rot": rot, "cols": 200}
        elif kind == "persons":
            c = {"kind": kind, "path": rng.choice(["tc", "tcg"]), "rows": _log(rng, 1000, 60000),
                 "queries": _log(rng, 4, 32), "rot": rot, "cols": 200}
        elif kind == "stage":
            c = {"kind": kind, "path": rng.choice(["tc", "tcg", "i8mma"]), "rows": _log(rng, 100, 16384),
                 "queries": _log(rng, 1, 32), "rot": rot, "cols": cols}
        elif kind == "compare":
            c = {"kind": kind, "rows": _log(rng, 1000, 65536), "queries": _log(rng, 1, 32), "rot": rot,
                 "mode": rng.choice(["lift", "lift", "plain", "const", "none"])}
        else:
            c = {"kind": kind, "rows": _log(rng, 64, 16384), "cols": cols, "ring": rng.choice([16, 16, 32])}
        if _cost(c) <= cap:
            return c


# ---------------------------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------------------------

def _geom(c):
    rot = c["rot"]
    return ipc.ipc_geom(16, c["cols"], 4, -(rot // 2), rot)


def _l(c):
    return 64 * c.get("cols", 200)


def _seeds(seed):
    return [0x51EED0 + 977 * seed + j for j in range(3)]


def _gen(seed, salt):
    g = torch.Generator(device="cuda")
    g.manual_seed(1000003 * seed + salt)
    return g


def _words(g, n, w):
    # the low 32 bits of two draws, so that all 64 bits of a word are used
    a = torch.randint(0, 1 << 32, (n, w), generator=g, device="cuda", dtype=torch.int64)
    b = torch.randint(0, 1 << 32, (n, w), generator=g, device="cuda", dtype=torch.int64)
    return a | (b << 32)


def _mask_words(g, n, w):
    # Bernoulli(231/256 = 0.902): one bit of the probability's binary expansion per draw, lowest first
    m = torch.zeros((n, w), dtype=torch.int64, device="cuda")
    for k in range(8):
        r = _words(g, n, w)
        m = (m | r) if (231 >> k) & 1 else (m & r)
    return m


def _unpack(words):
    return ((words[:, :, None] >> torch.arange(64, device="cuda")) & 1).reshape(words.shape[0], -1)


def _pack(bits):
    b = bits.reshape(bits.shape[0], -1, 64).to(torch.int64) << torch.arange(64, device="cuda")
    return b.sum(-1)


def _db_bits(c, seed, salt=0):
    g = _gen(seed, 1 + 16 * salt)
    return _words(g, c["rows"], _l(c) // 64), _mask_words(g, c["rows"], _l(c) // 64)


def _query_bits(c, seed, n, db, salt=0):
    """n query codes: every other one a near-duplicate of a database row, rotated within the range."""
    g = _gen(seed, 2 + 16 * salt)
    code, mask = _words(g, n, _l(c) // 64), _mask_words(g, n, _l(c) // 64)
    rows = torch.randint(0, c["rows"], (n,), generator=g, device="cuda").cpu().numpy()
    pick = torch.randint(0, 2, (n,), generator=g, device="cuda").cpu().numpy()
    flips = _unpack(_words(g, n, _l(c) // 64) & _words(g, n, _l(c) // 64) & _words(g, n, _l(c) // 64))
    geom = _geom(c)
    for q in np.nonzero(pick)[0]:
        r, s = int(rows[q]), geom.rot_lo + int(rows[q]) % geom.R
        cb, mb = _unpack(db[0][r:r + 1]), _unpack(db[1][r:r + 1])
        cb = cb ^ (flips[q:q + 1])
        roll = lambda b: torch.roll(b.reshape(1, 16, c["cols"], 4), -s, 2).reshape(1, -1)
        code[q], mask[q] = _pack(roll(cb))[0], _pack(roll(mb))[0]
    return code, mask


def _encode(c, bits, client_seed, side, path="tc", lift="mpc", plain=False):
    """A0: the three components (or Galois-ring shares) of code and mask, as a client computes them."""
    n, l = bits[0].shape[0], _l(c)
    code = torch.empty((3, n, l), dtype=torch.int16, device="cuda")
    mask = torch.empty_like(code)
    fn = ipc.ipc_encode_share_galois if path == "tcg" else ipc.ipc_encode_share
    fn(bits[0], bits[1], n, l, client_seed, side, 0, code, mask)
    if plain:
        m = torch.empty((n, l), dtype=torch.int16, device="cuda")
        ipc.ipc_encode_plain_mask(bits[1], n, l, m)
        return list(code), [m, None, None]
    if lift != "mpc":
        code32 = torch.empty((3, n, l), dtype=torch.int32, device="cuda")
        mask32 = torch.empty_like(code32)
        ipc.ipc_encode_share32(bits[0], bits[1], n, l, client_seed, side, 0, code32, mask32)
        return (list(code32) if lift == "none" else list(code)), list(mask32)
    return list(code), list(mask)


class _Context:
    """A loaded context, released with the state that holds it."""

    def __init__(self, c, seed, salt=0, max_queries=1, **cfg):
        self.ctx = ipc.ipc_create(ipc.make_config(_geom(c), thr_a=THR_A, path=c["path"], max_queries=max_queries,
                                                  seeds=_seeds(seed), **cfg))
        ipc.ipc_set_input_stream(self.ctx)
        self.db = _db_bits(c, seed, salt)
        kw = dict(path=c["path"], lift=cfg.get("lift", "mpc"), plain=cfg.get("plain_mask", False))
        for r0 in range(0, c["rows"], 16384):
            part = [b[r0:r0 + 16384].contiguous() for b in self.db]
            code, mask = _encode(c, part, DB_SEED + r0, 0, **kw)
            ipc.load_db_shares(self.ctx, code, mask, part[0].shape[0], 1)

    def __del__(self):
        if getattr(self, "ctx", None):
            ipc.ipc_destroy(self.ctx)
            self.ctx = None


def _hosted(vecs):
    return [None if v is None else v.cpu().pin_memory() for v in vecs]


def _request_queries(c, seed, db):
    """The raw bits of each request's queries."""
    return [_query_bits(c, seed, c["queries"], db, salt=i) for i in range(c["requests"])]


def _sizes(c):
    return [int(x) for x in c["sizes"].split(",")]


def prepare(case, seed):
    c = case
    st = {"case": c}
    if c["kind"] == "request":
        h = _Context(c, seed, max_queries=c["queries"], lift=c["lift"], plain_mask=c["plain"])
        st["queries"] = []
        for bits in _request_queries(c, seed, h.db):
            code, mask = _encode(c, bits, Q_SEED + seed, 1, c["path"], c["lift"], c["plain"])
            st["queries"].append((_hosted(code), _hosted(mask)) if c["host"] else (code, mask))
        st["holder"], h.db = h, None
    elif c["kind"] == "serve":
        sizes = _sizes(c)
        h = _Context(c, seed, max_queries=max(sizes))
        st["queries"] = []
        for i, n in enumerate(sizes):
            code, mask = _encode(c, _query_bits(c, seed, n, h.db, salt=i), Q_SEED + seed, 1, c["path"])
            st["queries"].append((_hosted(code), _hosted(mask), n))
        st["holder"], h.db = h, None
        torch.cuda.empty_cache()
        ipc.ipc_serve_start(h.ctx, pool_queries=sum(sizes))
    elif c["kind"] == "persons":
        hs = [_Context(c, seed, salt=e, max_queries=c["queries"]) for e in range(2)]
        enc = [_encode(c, _query_bits(c, seed, c["queries"], hs[e].db, salt=e), Q_SEED + seed, 1, c["path"])
               for e in range(2)]
        st["code"] = _hosted(enc[0][0] + enc[1][0])
        st["mask"] = _hosted(enc[0][1] + enc[1][1])
        st["holder"] = hs
        for h in hs:
            h.db = None
    elif c["kind"] == "stage":
        _prepare_stage(st, c, seed)
    elif c["kind"] == "compare":
        _prepare_compare(st, c, seed)
    else:
        st["bits"] = _db_bits(c, seed)
        n, l, dt = c["rows"], _l(c), torch.int16 if c["ring"] == 16 else torch.int32
        st["code"] = torch.empty((3, n, l), dtype=dt, device="cuda")
        st["mask"] = torch.empty_like(st["code"])
        st["planes"] = torch.empty((2, 3, c["ring"] // 8, n, l), dtype=torch.int8, device="cuda")
        st["seed"] = DB_SEED + seed
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    return st


def _tags(Q, R, req=7):
    t = torch.empty((Q * R, 2), dtype=torch.int32)
    n = torch.arange(Q * R)
    t[:, 0], t[:, 1] = req, ((n // R) << 5) | (n % R)
    return t.cuda()


def _roots_shape(c):
    return 3, c["queries"] * c["rot"], -(-c["rows"] // 1024)


def _prepare_stage(st, c, seed):
    n, l, Q, R = c["rows"], _l(c), c["queries"], c["rot"]
    db = _db_bits(c, seed)
    x = _encode(c, db, DB_SEED + seed, 0, c["path"])
    y = _encode(c, _query_bits(c, seed, Q, db), Q_SEED + seed, 1, c["path"])
    st["y"] = [torch.stack(v) for v in y]
    st["x"] = torch.empty((2, 3, 2, n, l), dtype=torch.int8, device="cuda")
    for v in range(2):
        for j in range(3):
            ipc.ipc_split_limbs(x[v][j], n * l, st["x"][v, j, 0], st["x"][v, j, 1])
    N = Q * R
    st["n_pad"], st["ldz"] = -(-N // 128) * 128, -(-n // 8) * 8
    K = l if c["path"] == "tcg" else 2 * l
    st["b"] = torch.empty((3, 2, 2, st["n_pad"], K), device="cuda",
                          dtype=torch.int8 if c["path"] == "i8mma" else torch.int16)
    st["z"] = torch.zeros((2, 3, N, st["ldz"]), dtype=torch.int16, device="cuda")
    st["roots"] = torch.zeros(_roots_shape(c), dtype=torch.int32, device="cuda")
    st["msb"] = torch.zeros((3, N, st["ldz"]), dtype=torch.uint8, device="cuda")
    st["bits"] = torch.zeros((3, Q), dtype=torch.uint8, device="cuda")
    st["tags"], st["geom"], st["seeds"] = _tags(Q, R), _geom(c), _seeds(seed)


def _compare_values(c, seed):
    """Plausible dot products and mask lengths of every (column, row): ml about 0.81 l, dot about 0, and a few
    matches among them."""
    g = _gen(seed, 5)
    N, n = c["queries"] * c["rot"], c["rows"]
    ml = 10368 + torch.randint(-150, 151, (N, n), generator=g, device="cuda", dtype=torch.int16)
    dot = torch.randint(-300, 301, (N, n), generator=g, device="cuda", dtype=torch.int16)
    hits = torch.rand((N, n), generator=g, device="cuda") < 0.02 / n
    return torch.where(hits, ml - 2000, dot), ml


def _split3(v, g, dt):
    """v as three uniformly random additive components of type dt."""
    top = 1 << (15 if dt == torch.int16 else 31)
    a, b = (torch.randint(-top, top, v.shape, generator=g, device="cuda", dtype=dt) for _ in range(2))
    return [a, b, v.to(dt) - a - b]


def _prepare_compare(st, c, seed):
    dot, ml = _compare_values(c, seed)
    g = _gen(seed, 6)
    pad = lambda v: torch.nn.functional.pad(v, (0, -c["rows"] % 8)).contiguous()
    dot, ml = pad(dot), pad(ml)
    mode = c["mode"]
    st["zc"] = _split3(dot, g, torch.int32 if mode == "none" else torch.int16)
    st["zm"] = ml if mode == "plain" else _split3(ml, g, torch.int16 if mode == "lift" else torch.int32)
    st["ldz"] = dot.shape[1]
    st["roots"] = torch.zeros(_roots_shape(c), dtype=torch.int32, device="cuda")
    st["bits"] = torch.zeros((3, c["queries"]), dtype=torch.uint8, device="cuda")
    st["tags"], st["seeds"] = _tags(c["queries"], c["rot"]), _seeds(seed)


# ---------------------------------------------------------------------------------------------
# One pass
# ---------------------------------------------------------------------------------------------

def _fetch(ctx, rid, n):
    shares = np.zeros((3, n), np.uint8)
    ipc.fetch_bit_shares(ctx, rid, shares, n)
    ipc.ipc_release(ctx, rid)
    return {"shares": shares, "bits": shares[0] ^ shares[1] ^ shares[2]}


def run(state):
    c = state["case"]
    kind = c["kind"]
    if kind == "request":
        ctx, src = state["holder"].ctx, 0 if c["host"] else 1
        ids = [ipc.submit_queries(ctx, code, mask, c["queries"], src) for code, mask in state["queries"]]
        return [_fetch(ctx, rid, c["queries"]) for rid in ids]
    if kind == "serve":
        ctx = state["holder"].ctx
        ids = [(ipc.ipc_serve_submit(ctx, code, mask, n), n) for code, mask, n in state["queries"]]
        return [_fetch(ctx, rid, n) for rid, n in ids]
    if kind == "persons":
        shares, _ = ipc.ipc_check_persons([h.ctx for h in state["holder"]], state["code"], state["mask"],
                                          c["queries"], 0)
        return {"shares": shares, "bits": shares[0] ^ shares[1] ^ shares[2]}
    if kind == "stage":
        return _run_stage(state, c)
    if kind == "compare":
        return _run_compare(state, c)
    n, l = c["rows"], _l(c)
    if c["ring"] == 16:
        ipc.ipc_encode_share(state["bits"][0], state["bits"][1], n, l, state["seed"], 0, 0, state["code"], state["mask"])
    else:
        ipc.ipc_encode_share32(state["bits"][0], state["bits"][1], n, l, state["seed"], 0, 0, state["code"],
                               state["mask"])
    for v, sh in enumerate((state["code"], state["mask"])):
        for j in range(3):
            p = state["planes"][v, j]
            if c["ring"] == 16:
                ipc.ipc_split_limbs(sh[j], n * l, p[0], p[1])
            else:
                ipc.ipc_split_limbs32(sh[j], n * l, list(p))
    return {"code": state["code"], "mask": state["mask"], "planes": state["planes"]}


def _run_stage(st, c):
    n, l, Q, N, path = c["rows"], _l(c), c["queries"], c["queries"] * c["rot"], c["path"]
    prep = {"tc": ipc.ipc_prep_query_f16, "tcg": ipc.ipc_prep_query_galois, "i8mma": ipc.ipc_prep_query}[path]
    for i in range(3):
        own, prev = st["seeds"][i], st["seeds"][(i + 2) % 3]
        for v in range(2):
            b, x, xp, z = st["b"][i, v], st["x"][v, i], st["x"][v, (i + 2) % 3], st["z"][v, i]
            prep(st["y"][v], Q, st["geom"], i, b[0], b[1], st["n_pad"])
            tail = (N, st["n_pad"], l, st["tags"], own, prev, v, z, st["ldz"], 0)
            if path == "tcg":
                ipc.ipc_ring_gemm_tc_galois(256, x[0], x[1], n, b[0], b[1], *tail)
            elif path == "tc":
                ipc.ipc_ring_gemm_tc([x[0], xp[0]], [x[1], xp[1]], n, b[0], b[1], *tail)
            else:
                ipc.ipc_ring_gemm(path, [x[0], xp[0]], [x[1], xp[1]], n, b[0], b[1], *tail)
    z, roots = st["z"], st["roots"]
    ipc.ipc_compare(list(z[0]), list(z[1]), st["ldz"], N, n, 0, st["tags"], st["seeds"], THR_A, 5, roots,
                    roots.shape[2], st["msb"], st["ldz"])
    blocks = roots.clone()  # ipc_or_finalize uses its input as scratch
    ipc.ipc_or_finalize(roots, roots.shape[2], roots.shape[2], 5, Q, c["rot"], st["tags"], st["seeds"], st["bits"])
    opened = st["bits"][0] ^ st["bits"][1] ^ st["bits"][2]
    return {"z": z, "roots": blocks, "msb": st["msb"], "shares": st["bits"], "bits": opened}


def _run_compare(st, c):
    n, Q, N, roots, mode = c["rows"], c["queries"], c["queries"] * c["rot"], st["roots"], c["mode"]
    tail = (st["ldz"], N, n, 0, st["tags"], st["seeds"], THR_A)
    if mode == "lift":
        ipc.ipc_compare(st["zc"], st["zm"], *tail, 5, roots, roots.shape[2])
    elif mode == "plain":
        ipc.ipc_compare_plain(st["zc"], st["zm"], *tail, 5, roots, roots.shape[2])
    else:
        z16, z32 = (None, st["zc"]) if mode == "none" else (st["zc"], None)
        ipc.ipc_compare_liftfree(z16, z32, st["zm"], *tail, 0, 5, roots, roots.shape[2])
    blocks = roots.clone()
    ipc.ipc_or_finalize(roots, roots.shape[2], roots.shape[2], 5, Q, c["rot"], st["tags"], st["seeds"], st["bits"])
    return {"roots": blocks, "shares": st["bits"], "bits": st["bits"][0] ^ st["bits"][1] ^ st["bits"][2]}


# ---------------------------------------------------------------------------------------------
# What a pass cannot do without
# ---------------------------------------------------------------------------------------------

def _gemm_work(c, rows, queries):
    """Shares read once, query shares read once; limb multiply-adds of the parties' dot products: per ring
    multiply-add 3 limb products over Z_2^16 and 10 over Z_2^32, K = 2 l replicated and l with Galois shares."""
    l, lift = _l(c), c.get("lift", "mpc")
    k = l if c["path"] == "tcg" else 2 * l
    elem = {"mpc": (2, 2), "const": (2, 4), "none": (4, 4)}[lift]
    mac = {2: 3, 4: 10}
    bytes_, macs = 3 * l * elem[0], 3 * k * mac[elem[0]]
    if c.get("plain"):
        bytes_, macs = bytes_ + 2 * l, macs + 3 * l
    else:
        bytes_, macs = bytes_ + 3 * l * elem[1], macs + 3 * k * mac[elem[1]]
    cols = queries * c["rot"]
    return bytes_ * (rows + queries) + 3 * queries, 2 * macs * rows * cols


def work(case):
    c = case
    if c["kind"] == "request":
        b, f = _gemm_work(c, c["rows"], c["queries"])
        return {"bytes": c["requests"] * b, "flops": c["requests"] * f}
    if c["kind"] == "serve":
        b, f = _gemm_work(c, c["rows"], sum(_sizes(c)))
        return {"bytes": b, "flops": f}
    if c["kind"] == "persons":
        b, f = _gemm_work(c, c["rows"], c["queries"])
        return {"bytes": 2 * b, "flops": 2 * f}
    if c["kind"] == "stage":
        b, f = _gemm_work(c, c["rows"], c["queries"])
        per = c["rows"] * c["queries"] * c["rot"]
        return {"bytes": b + (12 + 3) * per, "flops": f}  # z of six GEMMs and the MSB components are outputs
    if c["kind"] == "compare":
        per = {"lift": 12, "plain": 8, "const": 18, "none": 24}[c["mode"]]
        cells = c["rows"] * c["queries"] * c["rot"]
        # bit-sliced AND gates of the comparison, 32 cells a word, about 10 word operations a gate
        gates = {"lift": 94, "plain": 29, "const": 61, "none": 61}[c["mode"]]
        return {"bytes": per * cells, "flops": cells * gates * 10 / 32}
    n, l, e = c["rows"], _l(c), c["ring"] // 8
    return {"bytes": n * l // 4 + 2 * 3 * n * l * e * 2, "flops": 2 * n * l * 30}  # Philox: about 30 operations a value


# ---------------------------------------------------------------------------------------------
# Plain results
# ---------------------------------------------------------------------------------------------

def _match(c, q, db):
    """Alg. 1 on the raw bits: for each query, whether 4 dot > ml at some rotation and row. dot and ml are whole
    numbers of at most l <= 16384, which float32 products and sums give exactly."""
    geom = _geom(c)

    def values(bits):
        m = _unpack(bits[1]).float()
        return m - 2 * (_unpack(bits[0]).float() * m), m

    qc, qm = values(q)
    hit = torch.zeros(qc.shape[0], dtype=torch.bool, device="cuda")
    torch.backends.cuda.matmul.allow_tf32 = False
    roll = lambda v, s: torch.roll(v.reshape(-1, 16, c["cols"], 4), s, 2).reshape(v.shape)
    rolled = [torch.cat([roll(v, geom.rot_lo + r) for r in range(geom.R)]) for v in (qc, qm)]
    for r0 in range(0, db[0].shape[0], 4096):
        dc, dm = values([b[r0:r0 + 4096] for b in db])
        hit |= (4 * (rolled[0] @ dc.T) > rolled[1] @ dm.T).any(1).reshape(geom.R, -1).any(0)
    return hit.to(torch.uint8)


def _philox(c0, c1, c2, c3, seed):
    """Philox4x32-10 (Salmon et al., SC'11) on int64 tensors holding 32-bit counters."""
    x = [c0, c1, c2, c3]
    k0, k1 = seed & M32, (seed >> 32) & M32
    for _ in range(10):
        p, q = x[0] * 0xD2511F53, x[2] * 0xCD9E8D57
        x = [((q >> 32) & M32) ^ x[1] ^ k0, q & M32, ((p >> 32) & M32) ^ x[3] ^ k1, p & M32]
        k0, k1 = (k0 + 0x9E3779B9) & M32, (k1 + 0xBB67AE85) & M32
    return x


def _zero_share(c, N, seed):
    """F(seed) of every column and row as the ring GEMM draws it, and the vector number apart."""
    n, out = c["rows"], []
    tag = _tags(c["queries"], c["rot"]).to(torch.int64)
    g = torch.arange(-(-n // 8), device="cuda")[None, :]
    for v in range(2):
        w = _philox(g.expand(N, -1), tag[:, 1:2], tag[:, 0:1], torch.full_like(g, (2 << 24) | v), seed)
        half = torch.stack([h for word in w for h in (word & 0xFFFF, word >> 16)], -1)
        out.append(half.reshape(N, -1)[:, :n])
    return out


def _exact_z(c, seed):
    """The messages z[v][party] of the stage calls, by 64-bit arithmetic (replicated sharing)."""
    n, Q, R = c["rows"], c["queries"], c["rot"]
    geom = _geom(c)
    db = _db_bits(c, seed)
    x = _exact_encode(db, DB_SEED + seed, 0)
    y = _exact_encode(_query_bits(c, seed, Q, db), Q_SEED + seed, 1)
    s = _seeds(seed)
    F = [_zero_share(c, Q * R, k) for k in s]
    ldz = -(-n // 8) * 8
    z = torch.zeros((2, 3, Q * R, ldz), dtype=torch.int64, device="cuda")
    for v in range(2):
        for i in range(3):
            p = (i + 2) % 3
            a = torch.cat([x[v][i], x[v][p]], 1).double()
            rot = lambda t: torch.stack([torch.roll(t.reshape(Q, 16, c["cols"], 4), geom.rot_lo + r, 2).reshape(Q, -1)
                                         for r in range(R)], 1).reshape(Q * R, -1)
            b = torch.cat([rot((y[v][i] + y[v][p]) & 0xFFFF), rot(y[v][i])], 1)
            # two 8-bit halves of b, so that every sum stays below 2^53
            d = sum(((b >> k) & 0xFF).double() @ a.T * (1 << k) for k in (0, 8))
            z[v, i, :, :n] = d.to(torch.int64) + F[i][v] - F[p][v]
    return z.to(torch.int16)


def _exact_encode(bits, client_seed, side):
    """ipc_encode_share's components, [vector][component][n][l] of values in [0, 2^16)."""
    n = bits[0].shape[0]
    cb, mb = _unpack(bits[0]), _unpack(bits[1])
    l = cb.shape[1]
    e, r = torch.arange(l // 4, device="cuda")[None, :], torch.arange(n, device="cuda")[:, None]
    out = []
    for v, val in enumerate((mb - 2 * (cb & mb), mb)):
        w = torch.stack(_philox(e.expand(n, -1), r, torch.full_like(e, (side << 8) | v), torch.full_like(e, 1 << 24),
                                client_seed), -1).reshape(n, l)
        x0, x1 = w & 0xFFFF, w >> 16
        out.append([x0, x1, (val - x0 - x1) & 0xFFFF])
    return out


def exact(case, seed):
    c = case
    if c["kind"] == "request":
        db = _db_bits(c, seed)
        return [{"shares": None, "bits": _match(c, q, db)} for q in _request_queries(c, seed, db)]
    if c["kind"] == "serve":
        db = _db_bits(c, seed)
        return [{"shares": None, "bits": _match(c, _query_bits(c, seed, n, db, salt=i), db)}
                for i, n in enumerate(_sizes(c))]
    if c["kind"] == "persons":
        hit = torch.zeros(c["queries"], dtype=torch.uint8, device="cuda")
        for e in range(2):
            db = _db_bits(c, seed, e)
            q = _query_bits(c, seed, c["queries"], db, salt=e)
            hit |= _match(c, q, db)
            for p in range(1, c["queries"]):
                hit[p] |= _match(c, [b[p:p + 1] for b in q], [b[:p] for b in q])[0]
        return {"shares": None, "bits": hit}
    if c["kind"] == "stage":
        db = _db_bits(c, seed)
        bits = _match(c, _query_bits(c, seed, c["queries"], db), db)
        small = c["path"] != "tcg" and c["rows"] * c["queries"] * c["rot"] * _l(c) < 4e10
        return {"z": _exact_z(c, seed) if small else None, "roots": None, "msb": None, "shares": None, "bits": bits}
    if c["kind"] == "compare":
        dot, ml = _compare_values(c, seed)
        hit = (4 * dot.to(torch.int32) > ml.to(torch.int32)).any(1).reshape(c["queries"], -1).any(1)
        return {"roots": None, "shares": None, "bits": hit.to(torch.uint8)}
    if c["ring"] == 32:
        return None
    code, mask, planes = [], [], []
    for vec, (to, sh) in enumerate(zip((code, mask), _exact_encode(_db_bits(c, seed), DB_SEED + seed, 0))):
        to.extend(x.to(torch.int16) for x in sh)
        for x in sh:
            lo = x.to(torch.int8)
            planes += [lo, ((x - lo) >> 8).to(torch.int8)]
    shape = (2, 3, 2, c["rows"], _l(c))
    return {"code": torch.stack(code), "mask": torch.stack(mask), "planes": torch.stack(planes).reshape(shape)}
