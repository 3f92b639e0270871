"""Performance cases of libgfpdot: the products a program asks the library
for, each through its public entry point on device-resident operands.

A case is a dict of plain values with a "kind":

  dot        one dot product (gfp_dot)
  batch      uneven dot products over mixed moduli, through a batch plan
             (gfp_batch_plan_*) or in one shot (gfp_dot_batched)
  matvec     one dense matrix-vector product (gfp_matvec)
  wiedemann  the captured iteration x <- A x (gfp_matvec_iterate), or with
             the projection u^T A^t x (gfp_matvec_sequence)
  block      dense block product C = A B (gfp_matmul_block, or
             gfp_matmul_block_prepared for an A prepared once)
  csr        sparse-row block product (gfp_matmul_block_csr)
  gfq        dot product over GF(p^k) in the discrete-logarithm
             representation (gfp_gfq_dot)

Residues travel as int32 tensors holding the bits of the uint32 values, as
the binding takes them.  Values are uniform in [0, p), the distribution the
methods are used on (random vectors and matrices over the field).
"""
from __future__ import annotations

import math

import torch

from paper_cs_0404008_gb300 import gfpdot as g

PRIMES = (32749, 65521, 67108859, 2147483647, 4294967291)

# (p, k): coefficients f[0..k-1] of a primitive polynomial x^k + f[k-1] x^(k-1) + ... + f[0]
FIELDS = {
    (2, 8): (1, 0, 1, 1, 1, 0, 0, 0),
    (65521, 1): (17,),
    (5, 3): (2, 3, 0),
    (7, 4): (5, 3, 1, 0),
    (3, 10): (2, 1, 0, 1, 0, 0, 0, 0, 0, 0),
}

CHUNK = 1 << 26   # elements generated at a time (bounds the 64-bit temporaries)


def listed():
    return [
        # a round of short, uneven dot products over mixed moduli: the small requests a service
        # collects into one launch (bound by the launch and the latency of one pass)
        {"name": "batch_64_short", "kind": "batch", "pairs": 64, "lg_lo": 6, "lg_hi": 13, "plan": True},
        # one dot product of 2^20 terms over GF(65521): the library's plainest call
        {"name": "dot_2e20", "kind": "dot", "p": 65521, "n": 1 << 20},
        # 4096 uneven pairs of 2^8 to 2^20 terms over five moduli, planned once: bulk work
        {"name": "batch_4096", "kind": "batch", "pairs": 4096, "lg_lo": 8, "lg_hi": 20, "plan": True},
        # a matrix-vector product of the smallest side a service registers, over the largest modulus
        {"name": "matvec_1024", "kind": "matvec", "p": 4294967291, "rows": 1024, "cols": 1024, "pad": True},
        # a rectangular system as it comes: odd sides, rows packed without padding
        {"name": "matvec_9001x7003", "kind": "matvec", "p": 67108859, "rows": 9001, "cols": 7003, "pad": False},
        # the Wiedemann iteration: 64 products with one 32768 x 32768 matrix over GF(2^31 - 1)
        {"name": "wiedemann_32768", "kind": "wiedemann", "p": 2147483647, "n": 32768, "iters": 64, "project": False},
        # the block product of block methods: A used once as it is
        {"name": "block_16384", "kind": "block", "p": 65521, "m": 16384, "k": 16384, "nb": 64, "pad": True, "prepared": False},
        # the same with a resident A, prepared once for many products
        {"name": "block_16384_prepared", "kind": "block", "p": 65521, "m": 16384, "k": 16384, "nb": 64, "pad": True, "prepared": True},
        # a large-modulus block job of the serving mix at its largest size
        {"name": "block_8192_p32", "kind": "block", "p": 4294967291, "m": 8192, "k": 8192, "nb": 64, "pad": True, "prepared": False},
        # a mid-sized rectangular block product with odd sides and packed rows
        {"name": "block_3001x5003x40", "kind": "block", "p": 65521, "m": 3001, "k": 5003, "nb": 40, "pad": False, "prepared": False},
        # the sparse-row block product at 1 % density
        {"name": "csr_16384", "kind": "csr", "p": 65521, "m": 16384, "k": 16384, "nb": 64, "density": 0.01},
        # a long dot product over an odd-characteristic extension field (Zech additions)
        {"name": "gfq_3p10_2e27", "kind": "gfq", "p": 3, "k": 10, "n": 1 << 27},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["dot", "batch", "matvec", "wiedemann", "block", "block", "csr", "gfq"])
    p = rng.choice(PRIMES)
    if kind == "dot":
        return {"kind": kind, "p": p, "n": _log_int(rng, 1 << 10, 1 << 24)}
    if kind == "batch":
        lo = rng.randint(6, 10)
        return {"kind": kind, "pairs": _log_int(rng, 16, 4096), "lg_lo": lo, "lg_hi": rng.randint(lo + 3, 20),
                "plan": rng.random() < 0.7}
    if kind == "matvec":
        return {"kind": kind, "p": p, "rows": _log_int(rng, 256, 16384), "cols": _log_int(rng, 256, 16384),
                "pad": rng.random() < 0.6}
    if kind == "wiedemann":
        return {"kind": kind, "p": p, "n": _log_int(rng, 1024, 16384), "iters": rng.randint(8, 64),
                "project": rng.random() < 0.5}
    if kind == "block":
        return {"kind": kind, "p": p, "m": _log_int(rng, 256, 16384), "k": _log_int(rng, 256, 16384),
                "nb": rng.choice([8, 32, 64, 64, 64, rng.randint(4, 128)]), "pad": rng.random() < 0.7,
                "prepared": rng.random() < 0.4}
    if kind == "csr":
        return {"kind": kind, "p": p, "m": _log_int(rng, 256, 16384), "k": _log_int(rng, 256, 16384),
                "nb": rng.choice([16, 32, 64, 64, rng.randint(4, 96)]),
                "density": round(math.exp(rng.uniform(math.log(0.002), math.log(0.05))), 5)}
    fp, fk = rng.choice(sorted(FIELDS))
    return {"kind": kind, "p": fp, "k": fk, "n": _log_int(rng, 1 << 14, 1 << 27)}


# ---- inputs ----

def _uniform(p, n, seed, stream):
    """n residues uniform in [0, p), as the int32 bits of uint32 values."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed((int(seed) * 1000003 + stream) & 0x7FFFFFFFFFFFFFFF)
    out = torch.empty(n, dtype=torch.int32, device="cuda")
    for b in range(0, n, CHUNK):
        e = min(n, b + CHUNK)
        out[b:e] = torch.randint(0, p, (e - b,), dtype=torch.int64, device="cuda", generator=gen).to(torch.int32)
    return out


def _matrix(p, rows, cols, seed, stream, pad):
    """rows x cols residues; with pad, rows start on 16-byte boundaries."""
    a = _uniform(p, rows * cols, seed, stream).view(rows, cols)
    ld = (cols + 3) // 4 * 4
    if not pad or ld == cols:
        return a
    store = torch.zeros((rows, ld), dtype=torch.int32, device="cuda")
    store[:, :cols] = a
    return store[:, :cols]


def _batch_shapes(case, seed):
    """Lengths 2^U, U uniform in [lg_lo, lg_hi), moduli uniform over PRIMES;
    vectors start on 16-byte boundaries: (lengths, moduli, offsets, total)."""
    gen = torch.Generator()
    gen.manual_seed(int(seed) & 0x7FFFFFFFFFFFFFFF)
    u = torch.rand(case["pairs"], dtype=torch.float64, generator=gen)
    lens = torch.exp2(case["lg_lo"] + (case["lg_hi"] - case["lg_lo"]) * u).to(torch.int64).tolist()
    ps = [PRIMES[i] for i in torch.randint(0, len(PRIMES), (case["pairs"],), generator=gen).tolist()]
    off, total = [], 0
    for n in lens:
        off.append(total)
        total += (n + 3) // 4 * 4
    return lens, ps, off, total


# The shapes of a batch case are part of the case (drawn from its own numbers),
# its values are drawn from the seed.
def _batch(case, seed):
    lens, ps, off, total = _batch_shapes(case, case["pairs"] * 1009 + case["lg_lo"] * 31 + case["lg_hi"])
    modulus = torch.ones(total, dtype=torch.int64)
    for n, p, o in zip(lens, ps, off):
        modulus[o:o + n] = p
    modulus = modulus.cuda()
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed) & 0x7FFFFFFFFFFFFFFF)
    xy = []
    for _ in range(2):
        t = torch.empty(total, dtype=torch.int32, device="cuda")
        for b in range(0, total, CHUNK):
            e = min(total, b + CHUNK)
            w = torch.randint(0, 1 << 62, (e - b,), dtype=torch.int64, device="cuda", generator=gen)
            t[b:e] = (w % modulus[b:e]).to(torch.int32)
        xy.append(t)
    return lens, ps, off, xy[0], xy[1]


def _csr(case, seed):
    """Bernoulli(density) pattern per row, values uniform in [1, p)."""
    m, k, p = case["m"], case["k"], case["p"]
    gen = torch.Generator(device="cuda")
    gen.manual_seed((int(seed) * 1000003 + 7) & 0x7FFFFFFFFFFFFFFF)
    counts, cols = [], []
    step = max(1, CHUNK // k)
    for r in range(0, m, step):
        hit = torch.rand((min(step, m - r), k), device="cuda", generator=gen) < case["density"]
        counts.append(hit.sum(1))
        cols.append(hit.nonzero()[:, 1].to(torch.int32))
    row_ptr = torch.zeros(m + 1, dtype=torch.int64, device="cuda")
    row_ptr[1:] = torch.cumsum(torch.cat(counts), 0)
    col = torch.cat(cols)
    val = torch.randint(1, p, (max(1, col.numel()),), dtype=torch.int64, device="cuda", generator=gen).to(torch.int32)
    if col.numel() == 0:
        col = torch.zeros(1, dtype=torch.int32, device="cuda")
    return row_ptr.to(torch.int32), col, val


def _empty(*shape):
    return torch.empty(shape, dtype=torch.int32, device="cuda")


def prepare(case, seed):
    kind, p = case["kind"], case.get("p")
    s = {"case": case}
    if kind != "gfq":
        s["ctx"] = g.Context(0)
    if kind == "dot":
        s["x"], s["y"], s["out"] = _uniform(p, case["n"], seed, 0), _uniform(p, case["n"], seed, 1), _empty(1)
    elif kind == "batch":
        lens, ps, off, s["x"], s["y"] = _batch(case, seed)
        ax, ay = s["x"].data_ptr(), s["y"].data_ptr()
        s["pairs"] = [(q, ax + 4 * o, ay + 4 * o, n) for n, q, o in zip(lens, ps, off)]
        s["out"] = _empty(case["pairs"])
        if case["plan"]:
            s["plan"] = g.BatchPlan(s["ctx"], s["pairs"])
    elif kind == "matvec":
        s["A"] = _matrix(p, case["rows"], case["cols"], seed, 0, case["pad"])
        s["x"], s["y"] = _uniform(p, case["cols"], seed, 1), _empty(case["rows"])
    elif kind == "wiedemann":
        n = case["n"]
        s["A"] = _matrix(p, n, n, seed, 0, True)
        s["x"], s["Y"] = _uniform(p, n, seed, 1), _empty(case["iters"], n)
        if case["project"]:
            s["u"], s["seq"] = _uniform(p, n, seed, 2), _empty(case["iters"] + 1)
    elif kind == "block":
        A = _matrix(p, case["m"], case["k"], seed, 0, case["pad"])
        s["B"] = _matrix(p, case["k"], case["nb"], seed, 1, False)
        s["C"] = _empty(case["m"], case["nb"])
        if case["prepared"]:
            s["prep"] = g.BlockPrep(s["ctx"], p, A)
        else:
            s["A"] = A
    elif kind == "csr":
        s["row_ptr"], s["col"], s["val"] = _csr(case, seed)
        s["B"], s["C"] = _matrix(p, case["k"], case["nb"], seed, 1, False), _empty(case["m"], case["nb"])
    else:
        q, n = p ** case["k"], case["n"]
        s["field"] = g.Field(p, case["k"], FIELDS[(p, case["k"])])
        for i, name in enumerate(("x", "y")):
            s[name] = torch.empty(n, dtype=torch.int16, device="cuda")
            s["field"].to_log(_uniform(q, n, seed, i), s[name])
        s["out"] = torch.empty(1, dtype=torch.int16, device="cuda")
    return s


def run(s):
    case = s["case"]
    kind, p = case["kind"], case.get("p")
    if kind == "dot":
        return g.gfp_dot(s["ctx"], p, s["x"], s["y"], s["out"])
    if kind == "batch":
        return s["plan"].exec(s["out"]) if case["plan"] else g.gfp_dot_batched(s["ctx"], s["pairs"], s["out"])
    if kind == "matvec":
        return g.gfp_matvec(s["ctx"], p, s["A"], s["x"], s["y"])
    if kind == "wiedemann":
        if case["project"]:
            g.gfp_matvec_sequence(s["ctx"], p, s["A"], s["x"], s["u"], s["seq"], case["iters"], Y=s["Y"])
            return {"seq": s["seq"], "Y": s["Y"]}
        return g.gfp_matvec_iterate(s["ctx"], p, s["A"], s["x"], s["Y"], case["iters"])
    if kind == "block":
        if case["prepared"]:
            return s["prep"].matmul(s["ctx"], s["B"], s["C"])
        return g.gfp_matmul_block(s["ctx"], p, s["A"], s["B"], s["C"])
    if kind == "csr":
        return g.gfp_matmul_block_csr(s["ctx"], p, case["k"], s["row_ptr"], s["col"], s["val"], s["B"], s["C"])
    return s["field"].dot(s["x"], s["y"], s["out"])


def work(case):
    """Each input read once, each output written once (4-byte residues, 2-byte
    codes, 2 bytes an entry for a prepared A whose residues fit 16 bits, else
    4); two operations a multiply-add."""
    kind = case["kind"]
    if kind == "dot":
        return {"bytes": 8 * case["n"] + 4, "flops": 2 * case["n"]}
    if kind == "batch":
        lens = _batch_shapes(case, case["pairs"] * 1009 + case["lg_lo"] * 31 + case["lg_hi"])[0]
        return {"bytes": 8 * sum(lens) + 4 * len(lens), "flops": 2 * sum(lens)}
    if kind == "matvec":
        r, c = case["rows"], case["cols"]
        return {"bytes": 4 * (r * c + r + c), "flops": 2 * r * c}
    if kind == "wiedemann":
        n, t = case["n"], case["iters"]
        return {"bytes": 4 * t * (n * n + 2 * n), "flops": 2 * t * n * n}
    if kind == "block":
        m, k, nb = case["m"], case["k"], case["nb"]
        entry = 2 if case["prepared"] and case["p"] <= 65536 else 4
        return {"bytes": entry * m * k + 4 * (k * nb + m * nb), "flops": 2 * m * k * nb}
    if kind == "csr":
        m, k, nb = case["m"], case["k"], case["nb"]
        nnz = int(m * k * case["density"])
        return {"bytes": 8 * nnz + 4 * (m + 1) + 4 * (k * nb + m * nb), "flops": 2 * nnz * nb}
    return {"bytes": 4 * case["n"] + 2, "flops": 2 * case["n"]}


# ---- the same results in plain 64-bit arithmetic ----

def _wide(t):
    """uint32 bits in an int32 tensor -> int64 values."""
    return t.to(torch.int64) & 0xFFFFFFFF


def _limbs(t):
    """Values below 2^32 -> (high, low) 16-bit halves in float64."""
    w = _wide(t)
    return (w >> 16).double(), (w & 0xFFFF).double()


def _join(hh, mid, ll, p):
    """(hh 2^32 + mid 2^16 + ll) mod p for exact float64 integers below 2^53."""
    r = (hh.to(torch.int64) % p) * 65536
    r = (r + mid.to(torch.int64) % p) % p * 65536
    return (r + ll.to(torch.int64) % p) % p


def _matmul(A, B, p):
    """A B mod p (int64) for matrices of residues: 16-bit halves multiplied in
    float64, exact since 2^32 times at most 2^20 terms stays below 2^53."""
    bh, bl = _limbs(B)
    rows = []
    step = max(1, CHUNK // max(1, A.shape[1]))
    for r in range(0, A.shape[0], step):
        ah, al = _limbs(A[r:r + step])
        rows.append(_join(ah @ bh, ah @ bl + al @ bh, al @ bl, p))
    return torch.cat(rows)


def _dot(x, y, p):
    t = 0
    for b in range(0, x.numel(), 1 << 20):
        xh, xl = _limbs(x[b:b + (1 << 20)])
        yh, yl = _limbs(y[b:b + (1 << 20)])
        t = (t + int(_join(xh @ yh, xh @ yl + xl @ yh, xl @ yl, p))) % p
    return t


def _bits(t):
    return t.to(torch.int32)


def _gfq_dot(x, y, p, k, f):
    """Code of the dot product: coefficient products summed in float64 (exact),
    folded by x^k = -sum f_j x^j, and the logarithm found by walking x^e."""
    conv = [0] * (2 * k - 1)
    for b in range(0, x.numel(), 1 << 20):
        dx, dy = [], []
        for src, dst in ((x, dx), (y, dy)):
            v = _wide(src[b:b + (1 << 20)])
            for _ in range(k):
                dst.append((v % p).double())
                v = v // p
        prod = (torch.stack(dx) @ torch.stack(dy).T).to(torch.int64).tolist()
        for i in range(k):
            for j in range(k):
                conv[i + j] = (conv[i + j] + prod[i][j]) % p
    for d in range(2 * k - 2, k - 1, -1):
        for j in range(k):
            conv[d - k + j] = (conv[d - k + j] - conv[d] * f[j]) % p
    want, q = conv[:k], p ** k
    if not any(want):
        return 0
    c = [1] + [0] * (k - 1)
    for e in range(q - 1):
        if c == want:
            return e if e else q - 1
        top = c[k - 1]
        c = [((c[j - 1] if j else 0) - top * f[j]) % p for j in range(k)]
    raise ValueError("not a primitive polynomial")


def exact(case, seed):
    kind, p = case["kind"], case.get("p")
    if kind == "dot":
        t = _dot(_uniform(p, case["n"], seed, 0), _uniform(p, case["n"], seed, 1), p)
        return _bits(torch.tensor([t], device="cuda"))
    if kind == "batch":
        lens, ps, off, x, y = _batch(case, seed)
        return _bits(torch.tensor([_dot(x[o:o + n], y[o:o + n], q) for n, q, o in zip(lens, ps, off)], device="cuda"))
    if kind == "matvec":
        A = _matrix(p, case["rows"], case["cols"], seed, 0, False)
        return _bits(_matmul(A, _uniform(p, case["cols"], seed, 1).view(-1, 1), p).view(-1))
    if kind == "wiedemann":
        n = case["n"]
        A = _matrix(p, n, n, seed, 0, False)
        v, ys = _uniform(p, n, seed, 1), []
        seq = [] if case["project"] else None
        u = _uniform(p, n, seed, 2) if case["project"] else None
        for t in range(case["iters"] + 1):
            if seq is not None:
                seq.append(_dot(u, v, p))
            if t == case["iters"]:
                break
            v = _bits(_matmul(A, v.view(-1, 1), p).view(-1))
            ys.append(v)
        Y = torch.stack(ys)
        return Y if seq is None else {"seq": _bits(torch.tensor(seq, device="cuda")), "Y": Y}
    if kind == "block":
        A = _matrix(p, case["m"], case["k"], seed, 0, False)
        return _bits(_matmul(A, _matrix(p, case["k"], case["nb"], seed, 1, False), p))
    if kind == "csr":
        row_ptr, col, val = _csr(case, seed)
        m, k, p = case["m"], case["k"], case["p"]
        B = _matrix(p, k, case["nb"], seed, 1, False)
        rp = row_ptr.to(torch.int64)
        rows, step = [], max(1, CHUNK // k)
        for r in range(0, m, step):
            e = min(m, r + step)
            q0, q1 = int(rp[r]), int(rp[e])
            dense = torch.zeros((e - r, k), dtype=torch.int32, device="cuda")
            ri = torch.repeat_interleave(torch.arange(e - r, device="cuda"), rp[r + 1:e + 1] - rp[r:e])
            dense[ri, col[q0:q1].to(torch.int64)] = val[q0:q1]
            rows.append(_matmul(dense, B, p))
        return _bits(torch.cat(rows))
    q = p ** case["k"]
    x, y = _uniform(q, case["n"], seed, 0), _uniform(q, case["n"], seed, 1)
    code = _gfq_dot(x, y, p, case["k"], FIELDS[(p, case["k"])])
    return torch.tensor([code], device="cuda").to(torch.int16)
