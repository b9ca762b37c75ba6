"""What is timed: the calls a user of this framework makes, over the range in which they are made.

The rings and workload shapes are the framework's own presets (workloads.PRESETS: N = 2^13 with two
or three primes up to N = 2^16 with sixteen). A party holds a context with its keys and the launch
variants the autotuner picked, as train.py and the benchmark set it up, and calls

  ntt       Context.ntt_forward / ntt_inverse on a copy of a batch of RNS polynomials
  arith     the element-wise operations of a batch: add, sub, ciphertext x plaintext, exact rescale
  product   ciphertext x ciphertext with fused relinearisation and rescale
  rotate    a slot rotation (automorphism and key switch)
  rotsum    the in-block rotate-and-sum of an inner product (hoisted key switches)
  encrypt   the client's packing and encryption of one served request
  decrypt   the client's decryption of predicted-rating rows
  epoch     one encrypted SGD epoch over an encrypted CSR matrix
  serve     a server's loop over a few requests: submit, tick until done, poll, take

Ciphertext residues are uniform modulo their primes, so the operations on ciphertexts take uniform
residues; where a plaintext matters (encrypt, decrypt, epoch, serve) real ones are encrypted.
"""
import math

import numpy as np
import torch

from paper_2509_03024_gb300 import capi
from paper_2509_03024_gb300 import workloads as W

KEY_SEED = 20250903
LR, LAM = 0.005, 0.02
SERVED_ITEMS, SERVED_K, SERVED_STEPS = 3706, 16, 5   # the served workload's resident item factors


def listed():
    return [
        # the smallest transform call: two polynomials on the paper's N = 8192 ring, launch-bound
        {"name": "ntt_small", "kind": "ntt", "preset": "sweep32", "polys": 2},
        # a bulk conversion between coefficient and evaluation form on the widest ring
        {"name": "ntt_batch", "kind": "ntt", "preset": "served", "polys": 24},
        # the linear operations on an odd number of ciphertexts part-way down the chain
        {"name": "arith_batch", "kind": "arith", "preset": "batched", "count": 9, "level": 10},
        # one product on the small ring: the latency of an interactive computation (60/40-bit primes)
        {"name": "product_small", "kind": "product", "preset": "tiny", "count": 1, "level": 2},
        # the products of an epoch's launch set
        {"name": "product_batch", "kind": "product", "preset": "paper", "count": 64, "level": 7},
        # one rotation of one large ciphertext: latency of a key switch
        {"name": "rotate_one", "kind": "rotate", "preset": "served", "count": 1, "level": 12, "step": 32},
        # inner products of an odd batch, one level below the top as in an epoch (15 rotation keys)
        {"name": "rotate_sum_batch", "kind": "rotsum", "preset": "paper", "count": 33, "level": 6, "kp": 16},
        # a client's request: its factor in every block and its ratings, five ciphertexts
        {"name": "encrypt_request", "kind": "encrypt", "preset": "served", "nnz": 40},
        # a client reads its answer: the predicted ratings of 3706 items, four ciphertexts at level 1
        {"name": "decrypt_rows", "kind": "decrypt", "preset": "served", "count": 4, "level": 1},
        # the smallest epoch: 64 x 48 at 6 % density, k = 4
        {"name": "epoch_tiny", "kind": "epoch", "preset": "tiny", "users": 64, "items": 48, "ratings": 184, "k": 4,
         "level": 2},
        # the paper-scale epoch: 943 x 1682, 90 % of 100,000 ratings, k = 10
        {"name": "epoch_paper", "kind": "epoch", "preset": "paper", "users": 943, "items": 1682, "ratings": 90000,
         "k": 10, "level": 7},
        # a server's mixed load: requests arriving while others are in flight
        {"name": "serve_mix", "kind": "serve", "preset": "served", "requests": 6, "per_tick": 2, "nnz_most": 300},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["ntt", "arith", "product", "rotate", "rotsum", "encrypt", "decrypt", "epoch", "epoch", "epoch",
                       "serve"])
    if kind in ("encrypt", "serve"):
        case = {"kind": kind, "preset": "served"}
        if kind == "encrypt":
            case["nnz"] = _log_int(rng, 5, 300)
        else:
            case["requests"] = rng.randint(1, 8)
            case["per_tick"] = rng.randint(1, 4)
            case["nnz_most"] = _log_int(rng, 20, 400)
        return case
    if kind == "epoch":
        preset = rng.choice(["sweep32", "tiny", "t12", "paper", "batched"])
        users, items = _log_int(rng, 20, 900), _log_int(rng, 20, 1600)
        most = min(users * items // 4, 600 if preset == "batched" else 60000)
        return {"kind": kind, "preset": preset, "users": users, "items": items,
                "ratings": _log_int(rng, min(20, most), most), "k": rng.choice([3, 4, 8, 10]),
                "level": rng.randint(2, len(W.PRESETS[preset].data_bits) - 1)}
    preset = rng.choice(["sweep32", "tiny", "t12", "paper", "batched", "served", "large"])
    pre = W.PRESETS[preset]
    top = len(pre.data_bits) - 1
    most = {13: 300, 12: 300, 15: 70}.get(pre.log_n, 24)
    case = {"kind": kind, "preset": preset}
    if kind == "ntt":
        case["polys"] = _log_int(rng, 1, most)
        return case
    case["count"] = _log_int(rng, 1, most if kind != "decrypt" else 6)
    case["level"] = rng.randint(0 if kind in ("rotate", "rotsum", "decrypt") else 1, top)
    if kind == "rotate":
        case["step"] = rng.choice([1, -1, 7, 32, -16, 512])
    if kind == "rotsum":
        case["kp"] = rng.choice([2, 3, 4, 8, 16])
    if kind == "decrypt":
        case["level"] = rng.randint(1 if preset in ("paper", "batched", "served", "large") else 0, top)
    return case


# ------------------------------------------------------------------ inputs


def _context(case, seed, steps=()):
    ctx = capi.Context.from_preset(W.PRESETS[case["preset"]])
    ctx.keygen(KEY_SEED + seed, steps)
    ctx.autotune()
    return ctx


def _residues(ctx, count, parts, gen):
    """`count` ciphertext-shaped buffers of `parts` components, uniform modulo each limb's prime."""
    out = torch.empty((count, parts, ctx.top + 1, ctx.n), dtype=torch.int64, device="cuda")
    for i in range(ctx.top + 1):
        out[:, :, i] = torch.randint(0, ctx.primes[i], (count, parts, ctx.n), generator=gen, device="cuda")
    return out.reshape(-1)


def _at_level(ctx, buf, count, level, parts=2):
    """The limbs 0..level that make up the ciphertexts of a capacity-layout buffer."""
    return buf.view(count, parts, ctx.top + 1, ctx.n)[:, :, : level + 1]


def _ratings(case, seed):
    users, items, nnz = case["users"], case["items"], case["ratings"]
    if case["preset"] in ("paper", "batched") and nnz >= 4 * users:
        return W.movielens_like(users, items, nnz, 1.0, seed, min_per_user=min(20, nnz // users))
    return W.uniform_ratings(users, items, nnz / (users * items), seed)


def _predictions(ctx, count, seed):
    """Predicted ratings in every slot (1..5, fractional)."""
    return np.random.default_rng(seed).uniform(1.0, 5.0, (count, ctx.slots))


def _request(nnz, seed):
    rng = np.random.default_rng(seed)
    pop = np.arange(1, SERVED_ITEMS + 1, dtype=np.float64) ** -1.0
    items = np.sort(rng.choice(SERVED_ITEMS, size=nnz, replace=False, p=pop / pop.sum())).astype(np.int32)
    ratings = rng.choice(np.arange(1, 6), size=nnz, p=W.RATING_PROBS).astype(np.float64)
    return rng.normal(0.0, 0.1, size=SERVED_K), items, ratings


def prepare(case, seed):
    kind = case["kind"]
    gen = torch.Generator(device="cuda").manual_seed(1000 + seed)
    st = {"case": dict(case)}
    if kind == "ntt":
        ctx = _context(case, seed)
        n = case["polys"]
        st.update(ctx=ctx, a=_residues(ctx, n, 1, gen), b=_residues(ctx, n, 1, gen))
        st.update(fwd=torch.empty_like(st["a"]), inv=torch.empty_like(st["b"]))
    elif kind in ("arith", "product", "rotate", "rotsum"):
        steps = {"rotate": [case.get("step", 0)], "rotsum": list(range(1, case.get("kp", 1)))}.get(kind, ())
        ctx = _context(case, seed, steps)
        n = case["count"]
        st.update(ctx=ctx, a=_residues(ctx, n, 2, gen), out=ctx.empty_ct(n))
        if kind in ("arith", "product"):
            st["b"] = _residues(ctx, n, 2, gen)
        if kind == "arith":
            st.update(sub=ctx.empty_ct(n), mul=ctx.empty_ct(n), res=ctx.empty_ct(n))
            st["pt"] = torch.empty(ctx.n, dtype=torch.int64, device="cuda")
            ctx.encode(np.random.default_rng(seed).normal(0, 1, 500), st["pt"])
    elif kind == "encrypt":
        ctx = _context(case, seed)
        kp = 16
        n_vb = -(-SERVED_ITEMS // (ctx.slots // (2 * kp)))
        st.update(ctx=ctx, request=_request(case["nnz"], seed), nonce=(1 + seed) << 20, UR=ctx.empty_ct(1),
                  R=ctx.empty_ct(n_vb))
    elif kind == "decrypt":
        ctx = _context(case, seed)
        st.update(ctx=ctx, cts=[])
        for t, z in enumerate(_predictions(ctx, case["count"], seed)):
            ct = ctx.empty_ct()
            ctx.encrypt(z, case["level"], 7 + t, ct)
            st["cts"].append(ct)
    elif kind == "epoch":
        csr, k = _ratings(case, seed), case["k"]
        ctx = capi.Context.from_preset(W.PRESETS[case["preset"]])
        ctx.keygen(KEY_SEED + seed, ctx.mf_rotation_steps(k))
        ctx.autotune()
        plan = capi.MfPlan(ctx, csr.n, csr.m, k, csr.row_ptr, csr.col_idx, csr.vals)
        U, V = ctx.empty_ct(plan.n_ub), ctx.empty_ct(plan.n_vb)
        plan.encrypt_factors(0, W.init_factors(csr.n, k, seed + 100), U)
        plan.encrypt_factors(1, W.init_factors(csr.m, k, seed + 200), V)
        st.update(ctx=ctx, plan=plan, U0=U, V0=V, U=U.clone(), V=V.clone())
    elif kind == "serve":
        ctx = capi.Context.from_preset(W.PRESETS[case["preset"]])
        ctx.keygen(KEY_SEED + seed, ctx.serve_rotation_steps(SERVED_K))
        ctx.autotune()
        m, k, n = SERVED_ITEMS, SERVED_K, case["requests"]
        packing = capi.MfPlan(ctx, 1, m, k, [0, 1], [0], [1.0])   # gives the item factors' batch layout
        V = ctx.empty_ct(packing.n_vb)
        packing.encrypt_factors(1, W.init_factors(m, k, seed + 200, 0.3), V)
        rng = np.random.default_rng(seed)
        reqs = []
        for r in range(n):
            nnz = int(round(math.exp(rng.uniform(math.log(5), math.log(case["nnz_most"])))))
            u0, items, ratings = _request(nnz, seed * 1000 + r)
            UR, R = ctx.empty_ct(1), ctx.empty_ct(packing.n_vb)
            ctx.encrypt_request(m, k, u0, items, ratings, (1 + r) << 20, UR, R)
            reqs.append((items, UR.cpu().pin_memory(), R.cpu().pin_memory()))   # uploads come from the host
        server = capi.Server(ctx, V, m, k, SERVED_STEPS, LR, LAM, max_slots=n)
        outs = [torch.zeros(packing.n_vb * ctx.ct_words, dtype=torch.int64).pin_memory() for _ in range(n)]
        st.update(ctx=ctx, server=server, reqs=reqs, outs=outs, n_vb=packing.n_vb)
    return st


# ------------------------------------------------------------------ one pass


def run(st):
    case, ctx = st["case"], st["ctx"]
    kind = case["kind"]
    if kind == "ntt":
        n, limbs = case["polys"], ctx.top + 1
        st["fwd"].copy_(st["a"])           # the transforms work in place; the caller keeps its input
        ctx.ntt_forward(st["fwd"], n, limbs)
        st["inv"].copy_(st["b"])
        ctx.ntt_inverse(st["inv"], n, limbs)
        return [st["fwd"], st["inv"]]
    if kind == "arith":
        n, lv = case["count"], case["level"]
        ctx.add(st["a"], st["b"], st["out"], n, lv)
        ctx.sub(st["a"], st["b"], st["sub"], n, lv)
        ctx.mul_plain(st["a"], st["pt"], st["mul"], n, lv)
        ctx.rescale(st["a"], st["res"], n, lv)
        return [_at_level(ctx, st["out"], n, lv), _at_level(ctx, st["sub"], n, lv), _at_level(ctx, st["mul"], n, lv),
                _at_level(ctx, st["res"], n, lv - 1)]
    if kind == "product":
        n, lv = case["count"], case["level"]
        ctx.mul_relin_rescale(st["a"], st["b"], st["out"], n, lv)
        return [_at_level(ctx, st["out"], n, lv - 1)]
    if kind == "rotate":
        ctx.rotate(st["a"], st["out"], case["count"], case["level"], case["step"])
        return [_at_level(ctx, st["out"], case["count"], case["level"])]
    if kind == "rotsum":
        ctx.rotate_sum(st["a"], st["out"], case["count"], case["level"], case["kp"])
        return [_at_level(ctx, st["out"], case["count"], case["level"])]
    if kind == "encrypt":
        u0, items, ratings = st["request"]
        ctx.encrypt_request(SERVED_ITEMS, SERVED_K, u0, items, ratings, st["nonce"], st["UR"], st["R"])
        return [st["UR"], st["R"]]
    if kind == "decrypt":
        return [ctx.decrypt(ct, case["level"]) for ct in st["cts"]]
    if kind == "epoch":
        plan, lv = st["plan"], case["level"]
        st["U"].copy_(st["U0"])            # an epoch updates the factors in place
        st["V"].copy_(st["V0"])
        plan.sgd_epoch(st["U"], st["V"], lv, LR, LAM)
        return [_at_level(ctx, st["U"], plan.n_ub, lv - 2), _at_level(ctx, st["V"], plan.n_vb, lv - 2)]
    # serve: `per_tick` requests are admitted before every tick; every answer is taken as it is reported
    server, n = st["server"], case["requests"]
    nxt, left, levels = 0, n, [0] * n
    while left:
        for _ in range(case["per_tick"]):
            if nxt < n:
                items, UR, R = st["reqs"][nxt]
                server.submit(nxt, items, UR, R)
                nxt += 1
        server.tick()
        for rid in server.poll():
            levels[rid] = server.take(rid, st["outs"][rid])
            left -= 1
    return [_at_level(ctx, o, st["n_vb"], lv) for o, lv in zip(st["outs"], levels)]


# ------------------------------------------------------------------ what a pass cannot do without


class _Ring:
    """Words (8 bytes) and modular additions and multiplications of the ring operations."""

    def __init__(self, preset):
        pre = W.PRESETS[preset]
        self.n, self.log_n, self.alpha = 1 << pre.log_n, pre.log_n, len(pre.special_bits)
        self.limbs = len(pre.data_bits)

    def ntt(self, rows):                      # one multiplication and two additions per butterfly
        return rows * 3 * (self.n // 2) * self.log_n

    def dnum(self, level):
        return -(-(level + 1) // self.alpha)

    def key_words(self, level):
        return self.dnum(level) * 2 * (level + 1 + self.alpha) * self.n

    def mod_up(self, level):
        l1, ops, rows = level + 1, 0, 0
        for j in range(self.dnum(level)):
            cnt = min(self.alpha, l1 - j * self.alpha)
            rows += l1 + self.alpha - cnt
            ops += 2 * cnt * (l1 + self.alpha - cnt) * self.n
        return ops + self.ntt(l1 + rows)

    def inner(self, level, keys=1):
        return keys * 4 * self.dnum(level) * (level + 1 + self.alpha) * self.n

    def mod_down(self, level, out_limbs, sources):
        return self.ntt(2 * sources + 2 * out_limbs) + 2 * out_limbs * self.n * (2 * sources + 2)

    def switch(self, level, keys=1):
        return self.mod_up(level) + self.inner(level, keys) + self.mod_down(level, level + 1, self.alpha)

    def tensor(self, level):
        return 5 * (level + 1) * self.n

    def relin_rescale(self, level):
        return self.mod_up(level) + self.inner(level) + self.mod_down(level, level, self.alpha + 1)

    def rescale(self, level, parts=2):
        return parts * (self.ntt(level + 1) + 2 * level * self.n)


def work(case):
    r, kind = _Ring(case["preset"]), case["kind"]
    n = r.n
    if kind == "ntt":
        rows = case["polys"] * r.limbs
        return {"bytes": 8 * n * 4 * rows, "flops": 2 * r.ntt(rows)}
    if kind in ("arith", "product", "rotate", "rotsum"):
        c, lv = case["count"], case["level"]
        ct = 2 * (lv + 1) * n
        if kind == "arith":
            return {"bytes": 8 * (c * (2 * ct + 3 * ct + 2 * lv * n) + n),
                    "flops": c * (3 * ct + r.rescale(lv)) + r.ntt(lv + 1)}
        if kind == "product":
            return {"bytes": 8 * (c * (2 * ct + 2 * lv * n) + r.key_words(lv)),
                    "flops": c * (r.tensor(lv) + r.relin_rescale(lv))}
        keys = case["kp"] - 1 if kind == "rotsum" else 1
        return {"bytes": 8 * (c * 2 * ct + keys * r.key_words(lv)), "flops": c * r.switch(lv, keys)}
    if kind == "encrypt":
        # five messages of the request, each slot value times a cosine per coefficient
        cts, nz = 1 + 4, 2 * SERVED_K * (n // 2 // 32) + SERVED_K * case["nnz"]
        return {"bytes": 8 * (cts * 2 * r.limbs * n + 2 * r.limbs * n), "flops": 2 * nz * n + cts * r.ntt(3 * r.limbs)}
    if kind == "decrypt":
        limbs = min(case["level"], 1) + 1
        fft = 5 * n * r.log_n
        return {"bytes": 8 * case["count"] * (2 * limbs * n + n // 2), "flops": case["count"] * (r.ntt(limbs) + fft)}
    if kind == "epoch":
        csr, k, lv = _ratings(case, 0), case["k"], case["level"]
        lay = capi.mf_layout(n // 2, csr.n, csr.m, k, csr.row_ptr, csr.col_idx, csr.vals)
        groups, nodes, bins = len(lay["groups"]), len(lay["nodes"]), int(lay["n_bins"])
        kp = 1 << (k - 1).bit_length()
        blocks = (n // 2) // (2 * kp)
        batches = -(-csr.n // blocks) - (-csr.m // blocks)
        per_group = (r.tensor(lv) + r.relin_rescale(lv) + r.mod_up(lv - 1) + r.inner(lv - 1, kp - 1)
                     + r.mod_down(lv - 1, lv, r.alpha) + 2 * r.rescale(lv) + 2 * r.tensor(lv - 1))
        per_node = r.inner(lv) + r.mod_down(lv, lv + 1, r.alpha) + r.relin_rescale(lv - 1) + r.switch(lv - 2)
        return {"bytes": 8 * (bins * lv * n + batches * 2 * (lv + 1 + lv - 1) * n + kp * r.key_words(lv)),
                "flops": groups * per_group + nodes * per_node}
    # serve: per fold-in step the inner products of the rated batches (all four at most), the update and
    # the block sums; then the prediction over four batches
    ops, top, nb = 0, r.limbs - 1, 4
    for s in range(SERVED_STEPS + 1):
        lv = top - 2 * s
        ops += nb * (r.tensor(lv) + r.relin_rescale(lv) + r.switch(lv - 1, 15))
        if s < SERVED_STEPS:
            ops += nb * (r.rescale(lv) + r.tensor(lv - 1)) + r.relin_rescale(lv - 1) + 5 * r.switch(lv - 2, 3) + r.rescale(lv)
    req = case["requests"]
    words = req * ((1 + nb) * 2 * r.limbs * n + nb * 2 * 2 * n) + 30 * r.key_words(top) + nb * 2 * r.limbs * n
    return {"bytes": 8 * words, "flops": req * ops}


def exact(case, seed):
    """Decryption returns the encrypted slot values. Every other output is a residue, compared bit for bit."""
    if case["kind"] != "decrypt":
        return None
    slots = 1 << (W.PRESETS[case["preset"]].log_n - 1)
    return list(np.random.default_rng(seed).uniform(1.0, 5.0, (case["count"], slots)))
