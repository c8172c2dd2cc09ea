"""The work a PIR server has this library do, as cases that can be timed and compared.

A case names one call of the Python binding (paper_2604_04696_gb300.gpir) and its sizes. Inputs are uniform residues
(what NTT-form data and uniform RLWE masks look like); a program keeps the parameter set, the resident database and its
device buffers between calls, and so does a state here. Outputs are 32-bit residues, exact modulo each prime.

Kinds: "rowsel" (gpir_rowsel_batch), "multi" (gpir_rowsel_multi over several resident databases), "expand"
(gpir_expand_query), "coltor" (gpir_coltor) and "pir" (gpir_pir_batch, the three phases in one call).
"""

import torch

from paper_2604_04696_gb300 import gpir as g

#: The two largest primes below 2^28 that are 1 mod 8192: one per RNS limb.
PRIMES = (268369921, 268361729)
LOG_BASE = 22   # gadget base 2^22 of the two trees


def listed():
    return [
        # one query against a toy database: launch latency
        {"name": "rowsel_plain", "kind": "rowsel", "N": 2048, "L": 1, "D0": 16, "D1": 16, "B": 1},
        # the batch sweep's database (512 MiB): a lone query, a small batch, a full batch
        {"name": "rowsel_1", "kind": "rowsel", "N": 4096, "L": 2, "D0": 256, "D1": 64, "B": 1},
        {"name": "rowsel_8", "kind": "rowsel", "N": 4096, "L": 2, "D0": 256, "D1": 64, "B": 8},
        {"name": "rowsel_32", "kind": "rowsel", "N": 4096, "L": 2, "D0": 256, "D1": 64, "B": 32},
        # a database whose rows, columns and clients fill no tile
        {"name": "rowsel_ragged", "kind": "rowsel", "N": 4096, "L": 2, "D0": 500, "D1": 90, "B": 50},
        # the 4 GiB database at 128 clients: throughput
        {"name": "rowsel_4gib", "kind": "rowsel", "N": 4096, "L": 2, "D0": 1024, "D1": 128, "B": 128},
        # one mixed batch of the serving loop: three resident databases, uneven batches
        {"name": "multi_serving", "kind": "multi", "N": 4096, "L": 2, "D0": 256, "D1": 64, "B": 16,
         "D0b": 512, "D1b": 64, "Bb": 9, "D0c": 1024, "D1c": 128, "Bc": 3},
        # query expansion for 32 clients: 256 selection ciphertexts and 18 for the column bits
        {"name": "expand_32", "kind": "expand", "N": 4096, "L": 2, "J": 9, "n_out": 274, "B": 32},
        # the column tournament over 64 columns for 32 clients, and a small one-limb ring
        {"name": "coltor_32", "kind": "coltor", "N": 4096, "L": 2, "D1": 64, "B": 32},
        {"name": "coltor_small", "kind": "coltor", "N": 2048, "L": 1, "D1": 16, "B": 3},
        # a whole server step: the latency of one client, the throughput of 32
        {"name": "pir_1", "kind": "pir", "N": 4096, "L": 2, "D0": 256, "D1": 64, "J": 8, "B": 1},
        {"name": "pir_32", "kind": "pir", "N": 4096, "L": 2, "D0": 256, "D1": 64, "J": 8, "B": 32},
    ]


def _log_int(rng, lo, hi):
    """An integer of [lo, hi], even over the logarithm."""
    return min(hi, max(lo, round(lo * (hi / lo) ** rng.random())))


def draw(rng):
    kind = rng.choice(["rowsel", "rowsel", "rowsel", "multi", "expand", "expand", "coltor", "coltor", "pir"])
    N, L = (4096, 2) if rng.random() < 0.7 else (rng.choice([1024, 2048, 4096]), rng.choice([1, 2]))
    if kind == "rowsel":
        return {"kind": kind, "N": N, "L": L, "D0": _log_int(rng, 16, 600), "D1": _log_int(rng, 8, 128),
                "B": _log_int(rng, 1, 100)}
    if kind == "multi":
        c = {"kind": kind, "N": N, "L": L}
        for s in ("", "b", "c"):
            c.update({"D0" + s: _log_int(rng, 64, 500), "D1" + s: _log_int(rng, 16, 100), "B" + s: _log_int(rng, 1, 32)})
        return c
    if kind == "expand":
        J = rng.randint(4, 9)
        return {"kind": kind, "N": N, "L": L, "J": J, "n_out": rng.randint((1 << (J - 1)) + 1, 1 << J),
                "B": _log_int(rng, 1, 40)}
    if kind == "coltor":
        return {"kind": kind, "N": N, "L": L, "D1": 1 << rng.randint(3, 7), "B": _log_int(rng, 1, 40)}
    D0 = _log_int(rng, 32, 300)
    return {"kind": kind, "N": N, "L": L, "D0": D0, "D1": 1 << rng.randint(4, 6), "J": (D0 - 1).bit_length(),
            "B": _log_int(rng, 1, 32)}


def _digits(L):
    """Digits of base 2^22 that cover the modulus."""
    Q = 1
    for q in PRIMES[:L]:
        Q *= q
    return -(-(Q - 1).bit_length() // LOG_BASE)


def _uniform(gen, L, N, *shape):
    """Uniform residues [*shape][L][N], limb l below PRIMES[l], as the library's 32-bit words."""
    x = torch.empty(*shape, L, N, dtype=torch.int32, device="cuda")
    for l in range(L):
        x[..., l, :].random_(0, PRIMES[l], generator=gen)
    return x


def _inputs(case, seed):
    """The arrays a client or the database owner sends, by name; databases are drawn first."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    L, N, B, kind = case["L"], case["N"], case["B"], case["kind"]
    x, ell = {}, _digits(L)
    if kind in ("rowsel", "multi", "pir"):
        for s in ("", "b", "c") if kind == "multi" else ("",):
            x["db" + s] = _uniform(gen, L, N, case["D0" + s], case["D1" + s])
    if kind in ("rowsel", "multi"):
        for s in ("", "b", "c") if kind == "multi" else ("",):
            x["ct" + s] = _uniform(gen, L, N, case["B" + s], case["D0" + s], 2)
    if kind in ("expand", "pir"):
        x["query"] = _uniform(gen, L, N, B, 2)
        x["evk"] = _uniform(gen, L, N, B, case["J"], ell, 2)
    if kind == "coltor":
        x["ct"] = _uniform(gen, L, N, B, case["D1"], 2)
    if kind in ("coltor", "pir"):
        x["rgsw"] = _uniform(gen, L, N, B, case["D1"].bit_length() - 1, 2 * ell, 2)
    return x


class _Handles:
    """The parameter set and the resident databases of one program, freed with it."""

    def __init__(self, case):
        self.params = g.gpir_params_create(case["N"], list(PRIMES[:case["L"]]))
        self.dbs = []

    def upload(self, D0, D1, db):
        self.dbs.append(g.gpir_db_upload(self.params, D0, D1, db, True, 0, torch.cuda.current_stream()))
        return self.dbs[-1]

    def __del__(self):
        for h in self.dbs:
            g.gpir_db_free(h)
        g.gpir_params_destroy(self.params)


def prepare(case, seed):
    L, N, B, kind = case["L"], case["N"], case["B"], case["kind"]
    x = _inputs(case, seed)
    st = {"case": case, "h": _Handles(case)}

    def empty(*shape):
        return torch.empty(*shape, 2, L, N, dtype=torch.int32, device="cuda")

    for s in ("", "b", "c"):
        if "db" + s in x:
            st["db" + s] = st["h"].upload(case["D0" + s], case["D1" + s], x.pop("db" + s))
    st.update(x)
    if kind in ("rowsel", "multi"):
        for s in ("", "b", "c") if kind == "multi" else ("",):
            st["out" + s] = empty(case["B" + s], case["D1" + s])
    elif kind == "expand":
        st["out"] = empty(B, case["n_out"])
    elif kind == "coltor":
        st["out"] = empty(B)
    else:
        st.update(sel=empty(B, case["D0"]), rows=empty(B, case["D1"]), out=empty(B))
    if kind == "multi":
        st["jobs"] = [(st["db" + s], case["B" + s], st["ct" + s], st["out" + s]) for s in ("", "b", "c")]
    return st


def run(st):
    case, stream = st["case"], torch.cuda.current_stream()
    kind, B = case["kind"], case["B"]
    if kind == "rowsel":
        g.gpir_rowsel_batch(st["db"], B, st["ct"], st["out"], g.GPIR_PATH_AUTO, stream)
    elif kind == "multi":
        g.gpir_rowsel_multi(st["jobs"], g.GPIR_PATH_AUTO, stream)
        return [st["out"], st["outb"], st["outc"]]
    elif kind == "expand":
        g.gpir_expand_query(st["h"].params, B, case["J"], case["n_out"], st["query"], st["evk"], st["out"], stream)
    elif kind == "coltor":
        g.gpir_coltor(st["h"].params, B, case["D1"], st["ct"], st["rgsw"], st["out"], stream)
    else:
        g.gpir_pir_batch(st["db"], B, case["J"], st["query"], st["evk"], st["rgsw"], st["sel"], st["rows"], st["out"],
                         g.GPIR_PATH_AUTO, stream)
        return {"selection": st["sel"], "rows": st["rows"], "answer": st["out"]}
    return st["out"]


def work(case):
    """Bytes: every input read once, every output written once. Operations: a multiplication and an addition for each
    modular product of the matrix products, the transforms' butterflies and the key products."""
    L, N, B, kind = case["L"], case["N"], case["B"], case["kind"]
    poly, ell = L * N, _digits(L)
    butterflies = N // 2 * (N.bit_length() - 1)
    words = products = 0
    if kind in ("rowsel", "multi", "pir"):
        for s in ("", "b", "c") if kind == "multi" else ("",):
            D0, D1, b = case["D0" + s], case["D1" + s], case["B" + s]
            words += poly * (D0 * D1 + 2 * b * D1 + (2 * b * D0 if kind != "pir" else 0))
            products += poly * 2 * b * D0 * D1
    if kind in ("expand", "pir"):
        n_out = case["n_out"] if kind == "expand" else case["D0"]
        nodes = B * sum(min(1 << j, n_out) for j in range(case["J"]))
        words += 2 * poly * B * (1 + case["J"] * ell + n_out)
        products += nodes * L * ((1 + ell) * butterflies + (2 * ell + 2) * N)
    if kind in ("coltor", "pir"):
        D1 = case["D1"]
        words += 2 * poly * B * ((D1 if kind == "coltor" else 0) + (D1.bit_length() - 1) * 2 * ell + 1)
        products += B * (D1 - 1) * L * ((2 + 2 * ell) * butterflies + 4 * ell * N)
    return {"bytes": 4 * words, "flops": 2 * products}


# ---- the same in 64-bit integers, plainly -----------------------------------


def _primitive_root(n, q):
    """psi = g^((q - 1) / 2n), g the smallest generator mod q."""
    f, m, d = set(), q - 1, 2
    while d * d <= m:
        while m % d == 0:
            f.add(d)
            m //= d
        d += 1
    f |= {m} - {1}
    gen = next(x for x in range(2, q) if all(pow(x, (q - 1) // p, q) != 1 for p in f))
    return pow(gen, (q - 1) // (2 * n), q)


def _powers(w, n, q):
    p = torch.ones(1, dtype=torch.int64, device="cuda")
    while p.numel() < n:
        p = torch.cat([p, p * pow(w, p.numel(), q) % q])
    return p[:n]


def _dft(x, w, q):
    """X_s = sum_j x_j w^(js) mod q over the last axis."""
    y = x.unsqueeze(-1)   # [..., r, s]: the transform of the terms j = r (mod the extent of r)
    while y.shape[-2] > 1:
        h, m = y.shape[-2] // 2, y.shape[-1]
        e, o = y[..., :h, :], y[..., h:, :] * _powers(pow(w, h, q), m, q) % q
        y = torch.cat([(e + o) % q, (e - o) % q], dim=-1)
    return y[..., 0, :]


def _ntt(x, q):
    """A_s = sum_j a_j psi^((2s+1) j) mod q, natural order."""
    psi = _primitive_root(x.shape[-1], q)
    return _dft(x * _powers(psi, x.shape[-1], q) % q, psi * psi % q, q)


def _intt(x, q):
    n = x.shape[-1]
    inv = pow(_primitive_root(n, q), q - 2, q)
    return _dft(x, inv * inv % q, q) * _powers(inv, n, q) % q * pow(n, q - 2, q) % q


def _digit_transforms(a):
    """NTT-form polynomials [..., L, N] -> NTTs [..., L, N] of the balanced base-2^22 digits of their centred values."""
    L, ell = a.shape[-2], _digits(a.shape[-2])
    r = [_intt(a[..., l, :], PRIMES[l]) for l in range(L)]
    x, Q = r[0], PRIMES[0]
    if L == 2:
        x = x + Q * ((r[1] - r[0]) % PRIMES[1] * pow(PRIMES[0], -1, PRIMES[1]) % PRIMES[1])
        Q *= PRIMES[1]
    x = torch.where(x > Q // 2, x - Q, x)
    z = 1 << LOG_BASE
    for i in range(ell):
        d = x if i == ell - 1 else (x + z // 2) % z - z // 2
        x = (x - d) // z
        yield torch.stack([_ntt(d % q, q) for q in PRIMES[:L]], dim=-2)


def _moduli(L):
    return torch.tensor(PRIMES[:L], dtype=torch.int64, device="cuda").view(L, 1)


def _rowsel(ct, db):
    B, D0, L, D1 = ct.shape[0], ct.shape[1], ct.shape[-2], db.shape[1]
    out = torch.zeros(B, D1, 2, L, ct.shape[-1], dtype=torch.int64, device="cuda")
    for i in range(D0):   # each product is below 2^56: 64 of them fit
        out.addcmul_(ct[:, i].long().unsqueeze(1), db[i].long().unsqueeze(1))
        if i % 64 == 63 or i == D0 - 1:
            out %= _moduli(L)
    return out


def _expand(query, evk, J, n_out):
    L, N = query.shape[-2:]
    q, s = _moduli(L), torch.arange(N, device="cuda")
    c, key = query.long().unsqueeze(1), evk.long()
    for j in range(J):
        k = (N >> j) + 1
        tau = c[..., ((2 * s + 1) * k % (2 * N) - 1) // 2]
        t = torch.stack([torch.zeros_like(tau[:, :, 0]), tau[:, :, 1]], dim=2)
        for i, d in enumerate(_digit_transforms(tau[:, :, 0])):
            t = (t + d.unsqueeze(2) * key[:, j, i].unsqueeze(1)) % q
        mono = torch.stack([_powers(pow(_primitive_root(N, p), -1, p), 2 * N, p)[(2 * s + 1 << j) % (2 * N)]
                            for p in PRIMES[:L]])
        c = torch.cat([(c + t) % q, (c - t) % q * mono % q], dim=1)[:, :n_out]
    return c


def _coltor(ct, rgsw):
    q, ell, c, key = _moduli(ct.shape[-2]), _digits(ct.shape[-2]), ct.long(), rgsw.long()
    for st in range(key.shape[1]):
        lo = c[:, 0::2]
        diff, c = (c[:, 1::2] - lo) % q, lo
        for p in range(2):
            for i, d in enumerate(_digit_transforms(diff[:, :, p])):
                c = (c + d.unsqueeze(2) * key[:, st, p * ell + i].unsqueeze(1)) % q
    return c[:, 0]


def exact(case, seed):
    x, kind = _inputs(case, seed), case["kind"]
    if kind == "rowsel":
        return _rowsel(x["ct"], x["db"])
    if kind == "multi":
        return [_rowsel(x["ct" + s], x["db" + s]) for s in ("", "b", "c")]
    if kind == "expand":
        return _expand(x["query"], x["evk"], case["J"], case["n_out"])
    if kind == "coltor":
        return _coltor(x["ct"], x["rgsw"])
    sel = _expand(x["query"], x["evk"], case["J"], case["D0"])
    rows = _rowsel(sel, x["db"])
    return {"selection": sel, "rows": rows, "answer": _coltor(rows, x["rgsw"])}
