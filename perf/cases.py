"""The work users of this library have it do, as cases that can be timed.

A case is one call, or the short sequence of calls, that a program makes once it holds its
context, keys and model: a secure inference end to end (features in, leaf bits out) as graph
session or as separate calls, the server's part of one (query ciphertexts in, result ciphertext
out), and the ring operations under it.  ``prepare`` makes what the program holds, ``run`` is
one pass through the public functions of ``paper_2104_09583_gb300.copse``.  Forests and queries
are the seeded random ones of ``paper_2104_09583_gb300.synth``.  Every output is exact (bits,
or residues), so any two correct implementations return equal values.
"""
import numpy as np
import torch

from paper_2104_09583_gb300 import copse as K
from paper_2104_09583_gb300 import synth

_INFER = ("session", "calls", "server")


def _case(name, kind, log_n, bits, primes, dnum, trees=0, depth=0, complete=True, features=0, precision=0, classes=0,
          queries=0, encrypted=False, fused=False, g_r=0, g_l=0, polys=0, residues=0):
    return dict(name=name, kind=kind, log_n=log_n, bits=bits, primes=primes, dnum=dnum, trees=trees, depth=depth,
                complete=complete, features=features, precision=precision, classes=classes, queries=queries,
                encrypted=encrypted, fused=fused, g_r=g_r, g_l=g_l, polys=polys, residues=residues)


def listed():
    return [
        # one query of a small tree at the toy ring: the latency floor, all launches
        _case("toy_session", "session", 10, 50, 8, 3, 1, 3, True, 2, 4, 2, 1),
        # one query of a forest of about 100 branches, replayed as a graph: an interactive request
        _case("forest100_session", "session", 14, 55, 10, 4, 4, 5, False, 8, 8, 4, 1, g_r=64),
        # a queue of queries of that forest over four query ciphertexts, the last one part full, by
        # separate calls
        _case("forest100_calls", "calls", 14, 55, 10, 3, 4, 5, False, 8, 8, 4, 113, g_r=32, g_l=32),
        # 16-bit features on a small forest with the fused level products: many comparison products
        _case("prec16_session", "session", 14, 55, 11, 3, 2, 5, False, 2, 16, 3, 3, fused=True, g_r=8),
        # three forests of uneven size, 256 queries, in one graph launch (a batch from a queue)
        _case("batch3_session", "session", 14, 55, 10, 3, -3, 6, True, 32, 8, 4, 256, g_r=64, g_l=16),
        # the server's half for a large plaintext forest: two queries arrive encrypted, the encrypted
        # result goes back
        _case("forest64_server", "server", 15, 55, 10, 2, 64, 6, True, 16, 8, 4, 2, g_r=64, g_l=64),
        # an encrypted model: one query (latency), a few ciphertexts, and the batch it is made for
        _case("enc1_calls", "calls", 15, 55, 16, 3, 1, 6, True, 8, 16, 10, 1, True, g_r=32, g_l=32),
        _case("enc4_server", "server", 15, 55, 16, 3, 4, 6, True, 8, 16, 10, 160, True, g_r=80, g_l=64),
        _case("enc16_calls", "calls", 15, 55, 16, 3, 16, 6, True, 32, 16, 10, 128, True, g_r=128, g_l=128),
        # transforms both ways of a batch far larger than the cache
        _case("ntt_batch", "ntt", 15, 55, 16, 3, polys=64, residues=16),
        # one ring product at a small ring
        _case("product_small", "product", 12, 50, 4, 2, residues=3),
        # single ciphertext operations: product, rotation, modulus switch
        _case("ct_ops", "ops", 14, 55, 10, 3),
    ]


def _levels(precision, depth, fused):
    """Primes the circuit drops, and one to decrypt with."""
    lg = lambda x: max(x - 1, 0).bit_length()
    return (2 if fused else 3) + lg(precision) + lg(depth) + 1


def draw(rng):
    pick = lambda lo, hi: int(round(lo * (hi / lo) ** rng.random()))  # spread over the logarithm
    what = rng.choice(["toy", "forest", "forest", "multi", "server", "enc", "enc", "ntt", "product", "ops"])
    dnum = rng.choice([2, 3, 4])
    if what == "ntt":
        log_n, res = rng.choice([12, 13, 14, 15]), rng.randint(1, 16)
        return _drawn("ntt", log_n, rng.choice([50, 55]), 16, 3, polys=min(64, pick(1, 64)), residues=res)
    if what == "product":
        return _drawn("product", rng.choice([10, 11, 12, 13, 14, 15]), rng.choice([50, 55]), 16, 3,
                      residues=pick(1, 16))
    if what == "ops":
        return _drawn("ops", rng.choice([10, 12, 13, 14, 15]), rng.choice([50, 55]), rng.randint(4, 16), dnum)
    if what == "enc":
        trees, depth, p = pick(1, 12), rng.randint(2, 6), rng.choice([4, 8, 11, 16])
        primes = _levels(p, depth, False) + rng.randint(0, 3)
        return _drawn("calls" if rng.random() < 0.5 else "server", rng.choice([14, 15]), 55, primes, 3, trees, depth,
                      rng.random() < 0.5, pick(2, 32), p, 10, pick(1, 64), True, g_r=rng.choice([16, 48, 128]),
                      g_l=rng.choice([16, 64, 100]))
    fused = rng.random() < 0.3
    depth, p = rng.randint(2, 6), rng.choice([2, 5, 8, 16])
    trees = 1 if what == "toy" else pick(1, 16)
    log_n = rng.choice([10, 11, 12]) if what == "toy" else rng.choice([14, 15])
    if what == "toy":
        depth = min(depth, 4)
    primes = _levels(p, depth, fused) + rng.randint(0, 3)
    kind = {"toy": "session", "forest": "session", "multi": "calls", "server": "server"}[what]
    return _drawn(kind, log_n, rng.choice([50, 55]), primes, dnum, trees, depth, rng.random() < 0.5,
                  pick(2, 8) if what == "toy" else pick(2, 32), p, rng.randint(2, 10), pick(1, 8), False, fused,
                  rng.choice([8, 24, 64]), rng.choice([0, 16, 40]))


def _drawn(kind, *a, **k):
    c = _case("", kind, *a, **k)
    del c["name"]
    return c


# ---------------------------------------------------------------- inputs
def _forests(case, seed):
    """The case's forests as text with their queries, [(text, features array)]."""
    p, nf, nc = case["precision"], case["features"], case["classes"]
    if case["trees"] < 0:  # three forests of uneven size share the batch
        shapes = [(1, 3, True, 8, case["queries"] // 8), (4, 5, False, 16, 3 * case["queries"] // 8),
                  (16, 6, True, 32, case["queries"] // 2)]
    else:
        shapes = [(case["trees"], case["depth"], case["complete"], nf, case["queries"])]
    out = []
    for i, (nt, dp, comp, f, nq) in enumerate(shapes):
        # the trees' shapes belong to the case; what they compare, and their labels, to the seed
        text = synth.random_forest(17 * i + 5, nt, dp, f, p, nc, complete=comp)
        out.append((_redrawn(text, np.random.default_rng([seed, i]), f, p, nc),
                    synth.random_queries(77 * seed + i + 1, nq, f, p)))
    return out


def _redrawn(text, rng, features, precision, classes):
    toks = [line.split(" ") for line in text.strip().split("\n")]
    for t in toks[1:]:
        at = 0
        while at < len(t):
            if t[at] == "b":
                t[at + 1], t[at + 2] = str(rng.integers(features)), str(rng.integers(1 << precision))
                at += 3
            else:
                t[at + 1] = str(rng.integers(classes))
                at += 2
    return "\n".join(" ".join(t) for t in toks) + "\n"


class _Held:
    """What the program holds: handles, released in reverse order when it lets go of them."""

    def __init__(self):
        self._free = []

    def keep(self, handle, destroy):
        self._free.append((handle, destroy))
        return handle

    def __del__(self):
        while self._free:
            h, destroy = self._free.pop()
            destroy(h)


_CONTEXTS = {}


def _context(case):
    """A program's context for a ring and prime chain, made once."""
    key = (case["log_n"], case["bits"], case["primes"], case["dnum"])
    if key not in _CONTEXTS:
        _CONTEXTS[key] = K.copse_ctx_create(*key)
    return _CONTEXTS[key]


def _primes(case, ctx, n):
    return torch.tensor(K.copse_ctx_primes(ctx)[:n], dtype=torch.int64, device="cuda")


def _residues(rng, primes, polys, n):
    """Uniform residues [polys][prime][n] as 64-bit words on the device."""
    g = torch.Generator(device="cuda").manual_seed(int(rng.integers(1 << 40)))
    x = torch.randint(0, (1 << 62) - 1, (polys, len(primes), n), dtype=torch.int64, device="cuda", generator=g)
    return x.remainder_(primes.view(1, -1, 1))


def prepare(case, seed):
    s = _Held()
    s.kind, s.case, s.seed = case["kind"], case, seed
    s.ctx = ctx = _context(case)
    rng = np.random.default_rng(seed)
    if s.kind in _INFER:
        _prepare_inference(s, case, seed)
    elif s.kind == "ntt":
        s.x = _residues(rng, _primes(case, ctx, case["residues"]), case["polys"], 1 << case["log_n"])
    elif s.kind == "product":
        pr = _primes(case, ctx, case["residues"])
        s.a, s.b = (_residues(rng, pr, 1, 1 << case["log_n"])[0] for _ in range(2))
        s.c = torch.empty_like(s.a)
    else:
        # two ciphertexts, and the rotation keys of a small model's plan
        m = s.keep(K.copse_compile_forest(synth.random_forest(seed, 2, 3, 4, 4, 3), 4, 4, case["log_n"]),
                   K.copse_model_destroy)
        s.rot = K.copse_model_rotations(m)[0][-1]
        s.keys, s.evk = K.copse_keygen(ctx, 100 + seed, [m])
        s.keep(s.keys, K.copse_keys_destroy)
        s.keep(s.evk, K.copse_evk_destroy)
        s.ct = s.keep(K.copse_encrypt_features(ctx, s.keys, m, synth.random_queries(seed, 1, 4, 4), 7 + seed),
                      K.copse_ctbuf_destroy)
    torch.cuda.synchronize()
    return s


def _prepare_inference(s, case, seed):
    ctx, s.models, feats, s.nq, s.nout = s.ctx, [], [], [], []
    for text, q in _forests(case, seed):
        m = s.keep(K.copse_compile_forest(text, case["precision"], q.shape[1], case["log_n"]), K.copse_model_destroy)
        if case["encrypted"]:
            K.copse_model_set_encrypted(m, True)
        if case["fused"]:
            K.copse_model_set_fused(m, True)
        K.copse_model_set_bsgs(m, case["g_r"], case["g_l"])
        s.models.append(m)
        feats.append(torch.from_numpy(q.astype(np.int32)).reshape(-1))
        s.nq.append(len(q))
        s.nout.append(K.copse_model_info_get(m)["n_out"])
    s.feats = torch.cat(feats).cuda()
    s.keys, s.evk = K.copse_keygen(ctx, 100 + seed, s.models)
    s.keep(s.keys, K.copse_keys_destroy)
    s.keep(s.evk, K.copse_evk_destroy)
    if case["encrypted"]:
        K.copse_encrypt_model(ctx, s.keys, s.models[0], 9000 + seed)
    s.bits = torch.zeros(sum(n * o for n, o in zip(s.nq, s.nout)), dtype=torch.uint8, device="cuda")
    torch.cuda.synchronize()
    if s.kind == "session":
        # a model's queries fill as many ciphertexts (items of the graph) as they need
        items, counts = [], []
        for m, nq in zip(s.models, s.nq):
            i = K.copse_model_info_get(m)
            per = (1 << case["log_n"]) // (i["block"] * i["n_segments"])
            for q0 in range(0, nq, per):
                items.append(m)
                counts.append(min(per, nq - q0))
        s.session = s.keep(K.copse_session_create_batch(ctx, s.keys, s.evk, items, counts), K.copse_session_destroy)
        return
    # a resident model: the first inference of a program encodes it
    z = K.copse_encrypt_features(ctx, s.keys, s.models[0], np.zeros((0, case["features"]), np.uint32), 1)
    K.copse_ctbuf_destroy(K.copse_infer(ctx, s.evk, s.models[0], z))
    K.copse_ctbuf_destroy(z)
    if s.kind == "server":
        s.query = s.keep(K.copse_encrypt_features(ctx, s.keys, s.models[0], s.feats.data_ptr(), 50 + seed,
                                                  on_device=True, n_queries=s.nq[0]), K.copse_ctbuf_destroy)


# ---------------------------------------------------------------- one pass
def run(s):
    ctx, n = s.ctx, 1 << s.case["log_n"]
    stream = torch.cuda.current_stream().cuda_stream
    if s.kind == "session":
        K.copse_session_run(s.session, None, 50 + s.seed, stream=stream, feats_ptr=s.feats.data_ptr(),
                            out_ptr=s.bits.data_ptr())
        out, at = [], 0
        for q, o in zip(s.nq, s.nout):
            out.append(s.bits[at:at + q * o].view(q, o))
            at += q * o
        return out
    if s.kind == "calls":
        m = s.models[0]
        f = K.copse_encrypt_features(ctx, s.keys, m, s.feats.data_ptr(), 50 + s.seed, stream=stream, on_device=True,
                                     n_queries=s.nq[0])
        r = K.copse_infer(ctx, s.evk, m, f, stream=stream)
        K.copse_decrypt_labels(ctx, s.keys, m, r, s.nq[0], stream=stream, out_device_ptr=s.bits.data_ptr())
        K.copse_ctbuf_destroy(f)
        K.copse_ctbuf_destroy(r)
        return [s.bits.view(s.nq[0], s.nout[0])]
    if s.kind == "server":
        # the result ciphertexts in coefficient form, as they are sent back
        r = K.copse_infer(ctx, s.evk, s.models[0], s.query, stream=stream)
        out = [K.copse_ctbuf_export(ctx, r, i, n) for i in range(K.copse_ctbuf_count(r))]
        K.copse_ctbuf_destroy(r)
        return out
    if s.kind == "ntt":
        # to evaluation form, and a copy of that back
        fwd = s.x.clone()
        K.copse_ntt(ctx, fwd.data_ptr(), s.case["polys"], s.case["residues"], stream=stream)
        back = fwd.clone()
        K.copse_ntt(ctx, back.data_ptr(), s.case["polys"], s.case["residues"], inverse=True, stream=stream)
        return [fwd, back]
    if s.kind == "product":
        K.copse_poly_mul(ctx, s.a.data_ptr(), s.b.data_ptr(), s.c.data_ptr(), s.case["residues"], stream=stream)
        return [s.c]
    prod = K.copse_ct_mul(ctx, s.evk, s.ct, 0, s.ct, 1, stream=stream)
    rot = K.copse_ct_rotate(ctx, s.evk, s.ct, 2, s.rot, stream=stream)
    low = K.copse_ct_modswitch(ctx, s.ct, 3, stream=stream)
    out = [K.copse_ctbuf_export(ctx, b, 0, n) for b in (prod, rot, low)]
    for b in (prod, rot, low):
        K.copse_ctbuf_destroy(b)
    return out


# ---------------------------------------------------------------- what a pass cannot do without
def work(case):
    """Bytes: inputs, keys and model data read once, outputs written once.  Operations: two per
    modular multiply-add (one in each butterfly of a transform)."""
    n, lg = 1 << case["log_n"], case["log_n"]
    L, alpha = case["primes"], -(-case["primes"] // case["dnum"])
    bf = n // 2 * lg  # butterflies of one residue polynomial
    kind = case["kind"]
    if kind == "ntt":
        m = case["polys"] * case["residues"]
        return {"bytes": 4 * 8 * n * m, "flops": 2 * 2 * bf * m}
    if kind == "product":
        return {"bytes": 3 * 8 * n * case["residues"], "flops": 2 * (3 * bf + n) * case["residues"]}

    def switch(ell):  # one key switch at level ell: multiply-adds
        nd = -(-ell // alpha)
        return ell * bf + (nd * (ell + alpha) - ell) * bf + 2 * nd * (ell + alpha) * n + 2 * (alpha + ell) * bf

    def key(ell):
        return 8 * n * 2 * -(-ell // alpha) * (ell + alpha)

    if kind == "ops":
        macs = 2 * switch(L) + 4 * L * n + 2 * (2 * L) * bf + 2 * L * bf
        return {"bytes": 2 * key(L) + 8 * n * (8 * L + 2 * (3 * L - 2)), "flops": 2 * macs}
    byt = mac = 0
    for text, q in _forests(case, 0):
        m = K.copse_compile_forest(text, case["precision"], q.shape[1], lg)
        if case["encrypted"]:
            K.copse_model_set_encrypted(m, True)
        if case["fused"]:
            K.copse_model_set_fused(m, True)
        K.copse_model_set_bsgs(m, case["g_r"], case["g_l"])
        i = K.copse_model_info_get(m)
        K.copse_model_destroy(m)
        p, d, enc = case["precision"], i["depth"], case["encrypted"]
        lD = L - 1 - max(p - 1, 0).bit_length()
        lB = lD if case["fused"] else lD - 1
        cts = -(-len(q) // max(n // (i["block"] * i["n_segments"]), 1))
        diag = (0 if case["fused"] else i["q"] * lD) + d * min(i["n_leaves"], i["b"]) * lB // (1 if enc else d)
        prods = 2 * p - 3 + (p if enc else 0) + d - 1
        nr, nl = (0 if case["fused"] else i["n_rot_reshuffle"]), i["n_rot_level"]
        byt += 4 * q.size + len(q) * i["n_out"] + nr * key(lD) + nl * key(lB) + key(L) + 8 * n * diag
        if kind == "server":
            byt += cts * 8 * n * (2 * p * L + 2 * max(lB - 2, 1))
        else:
            mac += cts * p * 3 * L * bf
        mac += cts * (prods * switch((L + lD) // 2) + (4 if enc else 2) * n * diag)
        # hoisted rotations: the inner products; with an encrypted model every baby step is finished
        mac += cts * (nr * 2 * case["dnum"] * (lD + alpha) + nl * 2 * case["dnum"] * (lB + alpha)) * n
        if enc:
            mac += cts * (nr + nl) * 2 * (alpha + lB) * bf
    return {"bytes": byt, "flops": 2 * mac}


# ---------------------------------------------------------------- in plain numpy
def _walk(text, x):
    """Leaf bits of every query: the plain walk of each tree (feature < threshold goes right)."""
    cols = []
    for line in text.strip().split("\n")[1:]:
        toks, pos = line.split(), 0

        def node(reached):
            nonlocal pos
            if toks[pos] == "l":
                pos += 2
                cols.append(reached)
                return
            right = x[:, int(toks[pos + 1])] < int(toks[pos + 2])
            pos += 3
            node(reached & ~right)
            node(reached & right)

        node(np.ones(len(x), bool))
    return np.stack(cols, 1).astype(np.uint8)


def _negacyclic(a, b, q):
    """a b mod (X^n + 1, q) by one big-integer product (16 bytes a coefficient)."""
    n, w = len(a), 16
    pack = lambda v: int.from_bytes(np.stack([v, np.zeros_like(v)], 1).astype("<u8").tobytes(), "little")
    c = (pack(a) * pack(b)).to_bytes(2 * n * w, "little")
    c = [int.from_bytes(c[i * w:i * w + w], "little") % q for i in range(2 * n)]
    return np.array([(c[i] - c[i + n]) % q for i in range(n)], dtype=np.int64)


def exact(case, seed):
    if case["kind"] in ("session", "calls"):
        return [_walk(text, q) for text, q in _forests(case, seed)]
    if case["kind"] not in ("ntt", "product"):
        return None
    s = prepare(case, seed)
    if case["kind"] == "ntt":
        return [None, s.x.cpu().numpy()]
    if case["residues"] << case["log_n"] > 1 << 16:
        return None
    primes = K.copse_ctx_primes(s.ctx)
    a, b = s.a.cpu().numpy(), s.b.cpu().numpy()
    return [np.stack([_negacyclic(a[r], b[r], primes[r]) for r in range(len(a))])]
