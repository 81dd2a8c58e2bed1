"""The tcgen05 CRT kernel where its launch configurations change: one to four groups of 256 columns (with
three, two or one moduli side by side), a modulus count that the last tile does not fill, uneven
chunks with ragged row tiles, against the mma.sync kernel everywhere."""
import numpy as np
import pytest
import torch

from paper_2601_17561_gb300 import build as B
from paper_2601_17561_gb300 import engine as E
from paper_2601_17561_gb300 import icm as C
from paper_2601_17561_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def setup():
    B.build()
    # 56-bit primes: 17 CRT moduli
    eng = E.Engine(**{**E.TINY, "log_n_db": 7, "prime_bits": 56, "seed": 6}, hamming_weight=64).keygen()
    assert len(C.icm_ctx_crt_moduli(eng.ctx)) == 17
    W = synth.make_workload(n_eyes=34, n_db=231, seed=31)
    cuts = [0, 1, 150, 231]
    dbs = [eng.encrypt_db(W.db_codes[a:b], W.db_masks[a:b], chunk_id=i) for i, (a, b) in enumerate(zip(cuts, cuts[1:]))]
    return eng, W, dbs


@pytest.mark.parametrize("n_eyes", [1, 8, 9, 16, 17, 18, 24, 25, 34])
def test_column_groups(setup, n_eyes):
    eng, W, dbs = setup
    ct = eng.encrypt_query(W.q_codes[:n_eyes], W.q_masks[:n_eyes], W.eye_ids[:n_eyes])
    res = {}
    try:
        for v in (256, 1, 2, 3):
            C.icm_ctx_set_variant(eng.ctx, v)
            # columns just past a multiple of 256 (9, 17, 18, 25, 34 eyes) go to the digit planes on tcgen05
            outs = eng.match_batch(dbs, eng.prepare(ct, n_eyes, "f16_crt"))
            torch.cuda.synchronize()
            res[v] = [s.residues() for s in outs]
    finally:
        C.icm_ctx_set_variant(eng.ctx, 0)
    C.icm_device_status(True)
    for v in (1, 2, 3):
        for a, b in zip(res[v], res[256]):
            assert np.array_equal(a, b), v


@pytest.fixture(scope="module")
def wide():
    # 60-bit primes (18 CRT moduli), K = 2^14 + 2^7: an odd number of 16-word slabs over whole stages
    eng = E.Engine(log_n_db=7, log_n_q=7, n_limbs=2, n_limbs_q=1, prime_bits=60, log2_delta=40, seed=8,
                   hamming_weight=64).keygen()
    W = synth.make_workload(n_eyes=3, n_db=500, seed=33)
    cuts = [0, 3, 400, 500]
    dbs = [eng.encrypt_db(W.db_codes[a:b], W.db_masks[a:b], chunk_id=i) for i, (a, b) in enumerate(zip(cuts, cuts[1:]))]
    return eng, W, dbs


def _both(eng, dbs, ct, n_eyes):
    """Residues of the fp16 form on tcgen05 (digits up to 64 columns) and of the u64 form."""
    out = []
    for form in ("f16_crt", "u64"):
        s = eng.match_batch(dbs, eng.prepare(ct, n_eyes, form))
        torch.cuda.synchronize()
        out.append([x.residues() for x in s])
    C.icm_device_status(True)
    return out


@pytest.mark.parametrize("n_eyes,launches", [(1, 1), (2, 1), (3, 2)])
def test_few_columns(wide, n_eyes, launches):
    """31 and 62 columns multiply digits (one and two groups of 32 columns), 93 residues."""
    eng, W, dbs = wide
    assert C.icm_match_launches(eng.ctx, dbs[0].handle, n_eyes, C.FORMS["f16_crt"]) == launches
    ct = eng.encrypt_query(W.q_codes[:n_eyes], W.q_masks[:n_eyes], W.eye_ids[:n_eyes])
    a, b = _both(eng, dbs, ct, n_eyes)
    for x, y in zip(a, b):
        assert np.array_equal(x, y)


@pytest.mark.parametrize("sign", [1, -1])
def test_few_columns_extreme_digits(wide, sign):
    """Every database word and query coefficient at the value whose seven low digits are -128 (times
    the sign for the query): the first digits' products are all 2^14, the accumulators' bound."""
    eng, _, dbs = wide
    v = -sum(128 * 256 ** t for t in range(7))
    z = int.from_bytes(bytes([0x80] * 7 + [0]), "little")
    db = dbs[1]
    keep = db.buf.clone()
    try:
        db.buf.view(torch.int64).fill_(z)
        ct = torch.full((31 * eng.K,), (sign * v) % eng.primes[0], dtype=torch.int64, device=eng.device).view(torch.uint8)
        a, b = _both(eng, [db], ct, 1)
        assert np.array_equal(a[0], b[0])
        want = [(sign * v * v * eng.K) % q for q in eng.primes]
        assert all(np.all(a[0][l] == w) for l, w in enumerate(want))
    finally:
        db.buf.copy_(keep)


@pytest.mark.parametrize("M,N,K", [(1, 1, 2), (127, 31, 34), (129, 257, 1026), (64, 513, 48), (200, 769, 2080), (5, 1025, 96)])
def test_ppmm_canonical(M, N, K):
    """Canonical operands through the tcgen05 kernel (even K, 16-byte aligned) and, from an address that is
    only 8-byte aligned, through mma.sync: both equal to the u64 form."""
    q = [(1 << 60) - 93, (1 << 50) - 27, (1 << 31) - 1]
    g = torch.Generator(device="cuda").manual_seed(M + N + K)
    A = torch.stack([torch.randint(0, x, (M, K), generator=g, device="cuda", dtype=torch.int64) for x in q])
    Bm = torch.stack([torch.randint(0, x, (N, K), generator=g, device="cuda", dtype=torch.int64) for x in q])
    A[:, 0, :] = torch.tensor(q, device="cuda").view(-1, 1) - 1
    want = E.ppmm("u64", q, A, Bm)
    assert torch.equal(E.ppmm("f16_crt", q, A, Bm), want)
    shifted = torch.empty(A.numel() + 1, dtype=torch.int64, device="cuda")[1:].view(A.shape)
    shifted.copy_(A)
    assert shifted.data_ptr() % 16 == 8
    assert torch.equal(E.ppmm("f16_crt", q, shifted, Bm), want)


@pytest.mark.parametrize("n_eyes", [2, 8, 33, 34])
def test_match_host_in_one_part(setup, n_eyes):
    """icm_match_host with the workspace of twice the eyes (one part, where the columns share a round;
    34 eyes need two and stay in two parts) gives the same folded residues as with its own."""
    eng, W, dbs = setup
    h_ct = eng.encrypt_query(W.q_codes[:n_eyes], W.q_masks[:n_eyes], W.eye_ids[:n_eyes]).cpu().pin_memory()
    f, db, got = C.FORMS["f16_crt"], dbs[1], []
    for n in (n_eyes, 2 * n_eyes):
        wsb = C.icm_match_host_workspace_bytes(eng.ctx, db.handle, n, f)
        ws = torch.empty(wsb, dtype=torch.uint8, device=eng.device)
        h_fo = torch.zeros(eng.scores_bytes(db, n_eyes, True), dtype=torch.uint8).pin_memory()
        st = torch.cuda.Stream()
        C.icm_match_host(eng.ctx, db.handle, h_ct, n_eyes, f, h_fo, ws, wsb, stream=st)
        st.synchronize()
        got.append(h_fo)
    assert got[0].any() and torch.equal(got[0], got[1])


@pytest.fixture(scope="module")
def rows():
    # N_db = 2^11 on three limbs: the fewest rows beside which the last columns go to the digit planes
    eng = E.Engine(log_n_db=11, log_n_q=5, n_limbs=3, n_limbs_q=1, prime_bits=60, log2_delta=40, seed=8,
                   hamming_weight=16).keygen()
    W = synth.make_workload(n_eyes=40, n_db=300, seed=35)
    return eng, W, [eng.encrypt_db(W.db_codes[a:b], W.db_masks[a:b], chunk_id=i) for i, (a, b) in enumerate([(0, 3), (3, 300)])]


@pytest.mark.parametrize("n_eyes,launches", [(9, 3), (17, 3), (34, 3), (40, 4)])
def test_digits_beside_residues(rows, n_eyes, launches):
    """One, two and four groups of 256 columns as residues and the rest as digits (279, 527, 1,054 columns), and a
    second round of residues (1,240 columns), on the storage form: the residues of the mma.sync kernel."""
    eng, W, dbs = rows
    assert C.icm_match_launches(eng.ctx, dbs[1].handle, n_eyes, C.FORMS["f16_crt"]) == launches
    ct = eng.encrypt_query(W.q_codes[:n_eyes], W.q_masks[:n_eyes], W.eye_ids[:n_eyes])
    res = []
    try:
        for v in (256, 2):
            C.icm_ctx_set_variant(eng.ctx, v)
            outs = eng.match_batch(dbs, eng.prepare(ct, n_eyes, "f16_crt"))
            torch.cuda.synchronize()
            res.append([s.residues() for s in outs])
    finally:
        C.icm_ctx_set_variant(eng.ctx, 0)
    C.icm_device_status(True)
    for a, b in zip(*res):
        assert np.array_equal(a, b)


def _ppmm_operands(M, N, K):
    q = [(1 << 60) - 93, (1 << 50) - 27, (1 << 31) - 1]
    g = torch.Generator(device="cuda").manual_seed(M + N + K)
    A, Bm = (torch.stack([torch.randint(0, x, (n, K), generator=g, device="cuda", dtype=torch.int64) for x in q])
             for n in (M, N))
    return q, A, Bm


@pytest.mark.parametrize("M,N,K", [(1, 1, 192), (1, 1, 194), (100, 31, 192), (100, 31, 194), (300, 300, 2), (2000, 300, 2)])
def test_ppmm_short_products(M, N, K):
    """Both sides of the line between mma.sync and tcgen05 for short products, equal to the u64 form."""
    q, A, Bm = _ppmm_operands(M, N, K)
    assert torch.equal(E.ppmm("f16_crt", q, A, Bm), E.ppmm("u64", q, A, Bm))


def test_ppmm_short_product_time():
    """A short product of one wave takes the time that it takes with an odd K, which mma.sync computes (1.2 times it
    on tcgen05)."""
    B.build()
    t = {}
    for K in (63, 64):
        q, A, Bm = _ppmm_operands(300, 300, K)
        q, A, Bm = q[:1], A[:1].contiguous(), Bm[:1].contiguous()
        Cm = torch.empty((1, 300, 300), dtype=torch.int64, device="cuda")
        wb = C.icm_ppmm_workspace_bytes(C.FORMS["f16_crt"], 1, 300, 300, K)
        ws, ts = torch.empty(wb, dtype=torch.uint8, device="cuda"), []
        for _ in range(100):
            a, b = torch.cuda.Event(True), torch.cuda.Event(True)
            a.record()
            C.icm_ppmm(C.FORMS["f16_crt"], q, 1, A, Bm, Cm, 300, 300, K, ws, wb)
            b.record()
            torch.cuda.synchronize()
            ts.append(a.elapsed_time(b))
        t[K] = min(ts)
    assert t[64] < 1.15 * t[63]


@pytest.mark.parametrize("n_eyes", [1, 9, 40])
def test_variant_set_after_preparation(rows, n_eyes):
    """A query prepared under one variant gives the same residues under any other (its digit columns, if it has
    some, stay with the digit kernel)."""
    eng, W, dbs = rows
    ct = eng.encrypt_query(W.q_codes[:n_eyes], W.q_masks[:n_eyes], W.eye_ids[:n_eyes])
    res = []
    try:
        for prepare, match in [(256, 256), (2, 256), (2, 128), (2, 1), (256, 2), (256, 3)]:
            C.icm_ctx_set_variant(eng.ctx, prepare)
            q = eng.prepare(ct, n_eyes, "f16_crt")
            C.icm_ctx_set_variant(eng.ctx, match)
            outs = eng.match_batch(dbs, q)
            torch.cuda.synchronize()
            res.append([s.residues() for s in outs])
    finally:
        C.icm_ctx_set_variant(eng.ctx, 0)
    C.icm_device_status(True)
    for r in res[1:]:
        for a, b in zip(r, res[0]):
            assert np.array_equal(a, b)


def test_digit_kernel_bounded_wait_runs_out(wide):
    """The digit kernel's waits end by themselves: with a 20 ms bound and the query producers' copies withheld
    (test-only switch) it records ICM_ETIMEOUT and returns, the status is then clear, and the next launch is
    right."""
    eng, W, dbs = wide
    ct = eng.encrypt_query(W.q_codes[:1], W.q_masks[:1], W.eye_ids[:1])
    q, ref = eng.prepare(ct, 1, "f16_crt"), eng.match(dbs[1], eng.prepare(ct, 1, "u64"))
    assert C.icm_match_launches(eng.ctx, dbs[1].handle, 1, C.FORMS["f16_crt"]) == 1
    torch.cuda.synchronize()
    C.icm_device_status(True)
    C.icm_ctx_set_device_wait(eng.ctx, 20_000_000, True)
    try:
        eng.match(dbs[1], q)
        torch.cuda.synchronize()
    finally:
        C.icm_ctx_set_device_wait(eng.ctx, 0, False)
    with pytest.raises(C.IcmError) as e:
        C.icm_device_status(True)
    assert e.value.status == C.ICM_ETIMEOUT
    C.icm_device_status(True)
    s = eng.match(dbs[1], q)
    torch.cuda.synchronize()
    C.icm_device_status(True)
    assert np.array_equal(s.residues(), ref.residues())
