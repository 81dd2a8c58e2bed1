"""The work that a user of the library has it do, as timed cases.

Every case goes through the public entry points (engine.py over include/icm.h): matching passes of
one query batch against a resident encrypted database (query preparation, CCMM, fold) from one
eye on a door-sized database to 32 eyes on a full block at the paper's parameters, the plain
modular product, what happens to the scores afterwards (rescaling and fold, normalisation of
slot-encoded scores, decryption by the key holder), and the two encryptions (enrolment, query).
Sizes are those of the repository's workloads (engine.TINY / engine.PAPER, the command line's
slice, the batching benchmark) or lie between them; odd row and eye counts are among them.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2601_17561_gb300 import engine as E

CODE_BITS, CODE_BYTES, RHO = 12800, 1600, 31
D2 = 1 << 14


def listed():
    return [
        # a door: one eye, a small enrolled group, the small parameter set; latency of one pass
        dict(name="match_1_eye_256", kind="match", params="tiny", log_n_db=12, n_limbs=3, n_eyes=1, chunks="256",
             form="f16_crt"),
        # one eye at the paper's parameters (a checkpoint between batches, a quiet server)
        dict(name="match_1_eye_3000", kind="match", params="paper", log_n_db=12, n_limbs=8, n_eyes=1, chunks="3000",
             form="f16_crt"),
        # a partial batch against a database split in uneven chunks, one grouped pass
        dict(name="match_8_eyes_3_chunks", kind="match", params="paper", log_n_db=12, n_limbs=4, n_eyes=8,
             chunks="2457,3931,1843", form="f16_crt"),
        # an odd batch that is one column past 512
        dict(name="match_17_eyes_4095", kind="match", params="paper", log_n_db=12, n_limbs=8, n_eyes=17,
             chunks="4095", form="f16_crt"),
        # the headline: a full batch of 32 eyes, N_db = 2^14, eight primes, one full block
        dict(name="match_32_eyes_16384", kind="match", params="paper", log_n_db=14, n_limbs=8, n_eyes=32,
             chunks="16384", form="f16_crt"),
        # the plain u64 form on the small parameter set (4 eyes, 256 codes)
        dict(name="match_u64_4_eyes", kind="match", params="tiny", log_n_db=12, n_limbs=3, n_eyes=4, chunks="256",
             form="u64"),
        # the plain modular product on canonical residues of the caller's own matrices
        dict(name="ppmm_f16", kind="ppmm", n_limbs=3, m=3001, n=500, k=8192, form="f16_crt"),
        # what a server sends back: scores rescaled by Q' and folded
        dict(name="rescale_fold_32_eyes", kind="rescale_fold", log_n_db=12, n_limbs=8, n_eyes=32, n_db=3000),
        # slot-encoded scores multiplied by the inverse mask overlaps
        dict(name="normalize_slots_8_eyes", kind="normalize", log_n_db=13, n_limbs=4, n_eyes=8, n_db=4096),
        # the key holder decrypts a batch's scores
        dict(name="decrypt_8_eyes", kind="decrypt", log_n_db=12, n_limbs=8, n_eyes=8, n_db=3000),
        # enrolment: templates in host memory to an encrypted chunk in device memory
        dict(name="encrypt_db_1000", kind="encrypt_db", params="paper", log_n_db=12, n_limbs=4, n_db=1000),
        # a client's batch of query eyes: host templates to wire ciphertext
        dict(name="encrypt_query_32", kind="encrypt_query", log_n_db=12, n_limbs=8, n_eyes=32),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: any kind, sizes over the whole range of the listed ones."""
    kind = rng.choice(["match"] * 5 + ["ppmm", "rescale_fold", "normalize", "decrypt", "encrypt_db", "encrypt_query"])
    if kind == "match":
        params = rng.choice(["tiny", "paper", "paper"])
        form = rng.choice(["f16_crt"] * 4 + ["u64"])
        log_n_db = 12 if params == "tiny" else rng.choice([12, 12, 13, 14])
        n_limbs = 3 if params == "tiny" else rng.choice([2, 4, 6, 8])
        n_eyes = rng.randint(1, 4) if form == "u64" else _log_int(rng, 1, 32)
        hi = 400 if form == "u64" else 1 << log_n_db
        n_chunks = rng.choice([1, 1, 1, 2, 3]) if log_n_db == 12 and form != "u64" else 1
        if form == "u64":
            log_n_db, n_limbs = 12, min(n_limbs, 3 if params == "tiny" else 2)
        chunks = ",".join(str(_log_int(rng, 150, hi)) for _ in range(n_chunks))
        return dict(kind=kind, params=params, log_n_db=log_n_db, n_limbs=n_limbs, n_eyes=n_eyes, chunks=chunks, form=form)
    if kind == "ppmm":
        return dict(kind=kind, n_limbs=rng.randint(1, 4), m=_log_int(rng, 100, 5000), n=_log_int(rng, 20, 700),
                    k=_log_int(rng, 500, 8192), form=rng.choice(["f16_crt", "f16_crt", "u64"]))
    if kind in ("rescale_fold", "decrypt"):
        n_eyes = _log_int(rng, 1, 32) if kind == "rescale_fold" else _log_int(rng, 1, 8)
        return dict(kind=kind, log_n_db=rng.choice([12, 13]), n_limbs=rng.choice([4, 6, 8]), n_eyes=n_eyes,
                    n_db=_log_int(rng, 200, 4000))
    if kind == "normalize":
        return dict(kind=kind, log_n_db=rng.choice([11, 12, 13]), n_limbs=4, n_eyes=_log_int(rng, 1, 16),
                    n_db=_log_int(rng, 200, 4096))
    if kind == "encrypt_db":
        return dict(kind=kind, params=rng.choice(["tiny", "paper"]), log_n_db=12, n_limbs=rng.choice([2, 3, 4]),
                    n_db=_log_int(rng, 100, 5000))
    return dict(kind=kind, log_n_db=12, n_limbs=rng.choice([4, 8]), n_eyes=_log_int(rng, 1, 32))


# ------------------------------------------------------------------------------ inputs

def _engine_args(case, seed):
    if case.get("params", "paper") == "tiny":
        return dict(E.TINY, seed=seed)
    L = case["n_limbs"]
    # two query primes and Delta = 2^60 as in engine.PAPER; one and 2^40 where only two or three exist
    lq, delta = (2, 60) if L >= 4 else (1, 40)
    return dict(E.PAPER, log_n_db=case["log_n_db"], n_limbs=L, n_limbs_q=lq, log2_delta=delta, seed=seed)


def _shape(case):
    """(L, L_q, K, N_db) of a case with an engine."""
    a = _engine_args(case, 0)
    return a["n_limbs"], a["n_limbs_q"], D2 + (1 << a["log_n_q"]), 1 << a["log_n_db"]


def _rows(n, n_db, slots=False):
    """Stored rows of a chunk of n templates: the a-part, the full blocks, the last block's real rows
    and the tail coefficients that the fold reads."""
    if slots:
        return n_db + -(-n // (n_db // 2)) * n_db
    full, rem = divmod(n, n_db)
    m = n_db + full * n_db
    return m + (rem + n_db - max(rem, n_db - (RHO - 1)) if rem else 0)


def _pack(bits):
    w = (1 << torch.arange(8, device=bits.device, dtype=torch.int32))
    return (bits.view(bits.shape[0], -1, 8).to(torch.int32) * w).sum(-1).to(torch.uint8).cpu().numpy()


def _templates(n, seed):
    """Uniform iris codes and Bernoulli(0.9) masks, packed least significant bit first (host arrays)."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    codes, masks = [], []
    for i in range(0, n, 4096):
        m = min(4096, n - i)
        codes.append(_pack(torch.rand((m, CODE_BITS), generator=g, device="cuda") < 0.5))
        masks.append(_pack(torch.rand((m, CODE_BITS), generator=g, device="cuda") < 0.9))
    return np.concatenate(codes), np.concatenate(masks)


def _pair_templates(n_eyes, n_db, seed):
    """Query and database templates; every twentieth database row is a noisy copy of a query."""
    qc, qm = _templates(n_eyes, 4 * seed + 1)
    dc, dm = _templates(n_db, 4 * seed + 2)
    rng = np.random.default_rng(seed)
    for r in range(7, n_db, 20):
        flips = rng.integers(0, 256, (2, CODE_BYTES), dtype=np.uint8)
        dc[r] = qc[r % n_eyes] ^ (flips[0] & flips[1])
    return qc, qm, dc, dm


def _ids(n, seed):
    return np.arange(1, n + 1, dtype=np.uint64) + np.uint64(seed % (1 << 40)) * np.uint64(1 << 20)


def _odd_moduli(n):
    """Odd moduli below 2^60 (a caller's own), fixed."""
    return [(1 << 60) - 93 - 2 * 137 * i for i in range(n)]


def _residues(shape, q, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    return torch.stack([torch.randint(0, ql, shape, generator=g, device="cuda", dtype=torch.int64) for ql in q])


def prepare(case, seed):
    kind = case["kind"]
    if kind == "ppmm":
        q = _odd_moduli(case["n_limbs"])
        A = _residues((case["m"], case["k"]), q, 2 * seed + 1)
        B = _residues((case["n"], case["k"]), q, 2 * seed + 2)
        return dict(kind=kind, form=case["form"], q=q, A=A, B=B)
    eng = E.Engine(**_engine_args(case, seed % (1 << 31) + 1)).keygen()
    st = dict(kind=kind, eng=eng)
    if kind == "encrypt_query":
        st["codes"], st["masks"] = _templates(case["n_eyes"], 4 * seed + 1)
        st["ids"] = _ids(case["n_eyes"], seed)
        return st
    if kind == "encrypt_db":
        st["codes"], st["masks"] = _templates(case["n_db"], 4 * seed + 2)
        return st
    sizes = [int(x) for x in str(case["chunks"] if kind == "match" else case["n_db"]).split(",")]
    n = case["n_eyes"]
    qc, qm, dc, dm = _pair_templates(n, sum(sizes), seed)
    ct = eng.encrypt_query(qc, qm, _ids(n, seed))
    if kind == "normalize":
        db = eng.encrypt_db_slots(dc, dm, 16)
        st["scores"] = eng.rescale(eng.match(db, eng.prepare(ct, n, "f16_crt")))
        st["qm"], st["dm"] = torch.from_numpy(qm).cuda(), torch.from_numpy(dm).cuda()
        return st
    cuts = np.cumsum([0] + sizes)
    dbs = [eng.encrypt_db(dc[a:b], dm[a:b], chunk_id=i) for i, (a, b) in enumerate(zip(cuts[:-1], cuts[1:]))]
    if kind == "match":
        st.update(ct=ct, dbs=dbs, n_eyes=n, form=case["form"])
        return st
    # the database itself is not needed after the match: the scores are what the user holds
    st["scores"] = eng.match(dbs[0], eng.prepare(ct, n, "f16_crt"))
    st["scores"].db.buf = None
    return st


def _words(s):
    """Scores as the int64 view of their residues [L][columns][rows]."""
    L, n, M = s.shape
    return s.buf[: L * n * M * 8].view(torch.int64).view(L, n, M)


def run(state):
    kind = state["kind"]
    if kind == "ppmm":
        return E.ppmm(state["form"], state["q"], state["A"], state["B"])
    eng = state["eng"]
    if kind == "match":
        q = eng.prepare(state["ct"], state["n_eyes"], state["form"])
        if len(state["dbs"]) == 1:
            scores = [eng.match(state["dbs"][0], q)]
        else:
            scores = eng.match_batch(state["dbs"], q)
        folded = [eng.fold(s) for s in scores]
        return dict(scores=[_words(s) for s in scores], folded=[_words(f) for f in folded])
    if kind == "rescale_fold":
        r = eng.rescale(state["scores"])
        f = eng.fold(r)
        return dict(rescaled=_words(r), folded=_words(f))
    if kind == "normalize":
        out = eng.normalize(state["scores"], state["qm"], state["dm"], 36)
        return out.view(torch.int64)
    if kind == "decrypt":
        return eng.decrypt(state["scores"])
    if kind == "encrypt_db":
        db = eng.encrypt_db(state["codes"], state["masks"])
        return db.buf.view(torch.int64)
    ct = eng.encrypt_query(state["codes"], state["masks"], state["ids"])
    return ct.view(torch.int64)


# ------------------------------------------------------------------------------ work and exact values

def _mac_flops(bits, k):
    """Floating-point operations of one modular multiply-add of `bits`-bit residues over a depth k on
    8-bit exact tensor products: two per product, one product per 8 bits of the result's range."""
    return 2 * math.ceil((2 * bits + math.log2(max(k, 2))) / 8)


def work(case):
    kind = case["kind"]
    if kind == "ppmm":
        L, m, n, k = case["n_limbs"], case["m"], case["n"], case["k"]
        return dict(bytes=8 * L * (m * k + n * k + m * n), flops=_mac_flops(60, k) * L * m * n * k)
    L, Lq, K, N = _shape(case)
    bits = 50 if case.get("params") == "tiny" else 60
    cols = case.get("n_eyes", 0) * RHO
    groups = case.get("n_eyes", 0) * 2
    if kind == "match":
        M = sum(_rows(int(x), N) for x in str(case["chunks"]).split(","))
        return dict(bytes=8 * (Lq * cols * K + L * M * K + L * (cols + groups) * M),
                    flops=_mac_flops(bits, K) * L * M * cols * K)
    if kind == "encrypt_query":
        # one negacyclic product of degree N_q per (column, prime, block of the code): N log N butterflies
        return dict(bytes=2 * case["n_eyes"] * CODE_BYTES + 8 * Lq * cols * K, flops=10 * 13 * Lq * cols * K)
    M = _rows(case["n_db"], N, kind == "normalize")
    if kind == "encrypt_db":
        return dict(bytes=2 * case["n_db"] * CODE_BYTES + 8 * L * M * K, flops=10 * math.log2(N) * L * M * K)
    if kind == "rescale_fold":
        return dict(bytes=8 * ((L + Lq) * cols * M + Lq * groups * M), flops=10 * (L + 1) * (Lq + 1) * cols * M)
    if kind == "decrypt":
        return dict(bytes=8 * L * cols * M + 8 * cols * case["n_db"], flops=10 * math.log2(N) * L * cols * M)
    blocks = M // N - 1
    out = 2 * Lq * cols * blocks * N
    return dict(bytes=8 * (Lq * cols * M + out) + CODE_BYTES * case["n_db"], flops=10 * math.log2(N) * 1.5 * out)


def _unpack(t):
    return np.unpackbits(t, axis=1, bitorder="little")[:, :CODE_BITS]


def _exact_product(A, B, q):
    """A B^T modulo q (int64 residues): 20-bit parts, exact float64 products, Horner in base 2^20."""
    parts = [[((X >> (20 * i)) & 0xFFFFF).double() for i in range(3)] for X in (A, B)]
    mod = np.uint64(q)
    acc = np.zeros((B.shape[0], A.shape[0]), np.uint64)
    for s in range(4, -1, -1):
        t = sum(parts[1][s - i] @ parts[0][i].T for i in range(3) if 0 <= s - i < 3)
        for _ in range(5):
            acc = (acc << np.uint64(4)) % mod
        acc = (acc + t.cpu().numpy().astype(np.uint64) % mod) % mod
    return acc.astype(np.int64)


def exact(case, seed):
    """The decrypted numerators are the cleartext inner products of the masked bit-vectors, the plain
    product is a product of integers; the ciphertexts depend on the library's own random streams."""
    if case["kind"] == "ppmm" and case["k"] <= 8192:
        st = prepare(case, seed)
        return torch.from_numpy(np.stack([_exact_product(st["A"][i], st["B"][i], q) for i, q in enumerate(st["q"])]))
    if case["kind"] == "decrypt":
        qc, qm, dc, dm = _pair_templates(case["n_eyes"], case["n_db"], seed)
        c, m = _unpack(qc).reshape(-1, 16, 200, 4), _unpack(qm).reshape(-1, 16, 200, 4)
        rot = [np.stack([np.roll(x, -(r - RHO // 2), axis=2) for r in range(RHO)], 1).reshape(-1, CODE_BITS) for x in (c, m)]
        vec = [torch.from_numpy(((1 - 2 * a.astype(np.int32)) * b).astype(np.float32)).cuda().double()
               for a, b in (rot, (_unpack(dc), _unpack(dm)))]
        return (vec[0] @ vec[1].T).round().to(torch.int64)
    return None
