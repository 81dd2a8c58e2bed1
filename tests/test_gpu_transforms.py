"""The encryption kernels' products by the secrets (negacyclic transforms) at the edges of their range: the
smallest rings, one, two and four columns per block, partial blocks, two query primes, against the
oracle bit by bit."""
import threading

import numpy as np
import pytest
import torch

import oracle as O
from paper_2601_17561_gb300 import build as B
from paper_2601_17561_gb300 import engine as E
from paper_2601_17561_gb300 import synth

pytestmark = pytest.mark.gpu

# (log N_db, log N_q, limbs, query limbs, templates, eyes): N_db = 32 with rho = 31 and several blocks; sizes
# that leave one transform level over a multiple of three, two and none; N_q = 2^14 (one column per block)
SHAPES = [(5, 5, 2, 1, 70, 1), (7, 14, 3, 1, 300, 2), (9, 9, 2, 1, 40, 12), (11, 13, 4, 2, 30, 6)]


def _u64(t, shape):
    n = int(np.prod(shape))
    return t[: n * 8].view(torch.int64).cpu().numpy().view(np.uint64).reshape(shape)


def _from_digit_form(z, q):
    B8 = np.uint64(0x8080808080808080)
    c = ((z ^ B8) - B8).view(np.int64)
    return np.stack([np.where(c[i] < 0, c[i] + np.int64(ql), c[i]).view(np.uint64) for i, ql in enumerate(q)])


@pytest.mark.parametrize("log_n_db,log_n_q,L,Lq,n_db,n_eyes", SHAPES)
def test_encryption_ring_edges(log_n_db, log_n_q, L, Lq, n_db, n_eyes):
    B.build()
    prm = dict(log_n_db=log_n_db, log_n_q=log_n_q, n_limbs=L, n_limbs_q=Lq, prime_bits=60,
               log2_delta=60 if Lq == 2 else 40, seed=9)
    P = O.Params(**prm, h=16)
    W = synth.make_workload(n_eyes=n_eyes, n_db=n_db, seed=21)
    eng = E.Engine(**prm, hamming_weight=16).keygen()
    ct = O.query_encrypt(P, W.q_codes, W.q_masks, W.eye_ids)
    assert np.array_equal(_u64(eng.encrypt_query(W.q_codes, W.q_masks, W.eye_ids), ct.shape), ct)
    A = O.db_rows(P, W.db_codes, W.db_masks, O.db_layout(n_db, P.ndb, P.rho))
    db = eng.encrypt_db(W.db_codes, W.db_masks)
    assert np.array_equal(_from_digit_form(_u64(db.buf, A.shape), P.q), A)


@pytest.mark.parametrize("log_n_db,log_n_q,L,Lq,n_db,n_eyes", SHAPES)
def test_decryption_ring_edges(log_n_db, log_n_q, L, Lq, n_db, n_eyes):
    """Decryption (one cluster of L blocks per column, several b-blocks, a partial last one) gives the
    cleartext inner products exactly, at the full level and after the rescaling."""
    B.build()
    prm = dict(log_n_db=log_n_db, log_n_q=log_n_q, n_limbs=L, n_limbs_q=Lq, prime_bits=60,
               log2_delta=60 if Lq == 2 else 40, seed=9)
    W = synth.make_workload(n_eyes=n_eyes, n_db=n_db, seed=21)
    eng = E.Engine(**prm, hamming_weight=16).keygen()
    db = eng.encrypt_db(W.db_codes, W.db_masks)
    s = eng.match(db, eng.prepare(eng.encrypt_query(W.q_codes, W.q_masks, W.eye_ids), n_eyes, "u64"))
    rc, rm = O.rotated_templates(W.q_codes, W.q_masks, eng.rho)
    want = O.inner_from_counts(*O.hd_counts(rc, rm, O.unpack(W.db_codes), O.unpack(W.db_masks)))
    assert np.array_equal(eng.decrypt(s).cpu().numpy(), want)
    assert np.array_equal(eng.decrypt(eng.rescale(s)).cpu().numpy(), want)


@pytest.mark.parametrize("log_n_db,n_db", [(13, 50), (13, 8250), (14, 50), (14, 16440)])
def test_decryption_large_rings(log_n_db, n_db):
    """The block shapes of the larger rings, with one b-block and with a second, partial one."""
    B.build()
    prm = dict(log_n_db=log_n_db, log_n_q=9, n_limbs=2, n_limbs_q=1, prime_bits=60, log2_delta=40, seed=9)
    W = synth.make_workload(n_eyes=1, n_db=n_db, seed=21)
    eng = E.Engine(**prm, hamming_weight=16).keygen()
    db = eng.encrypt_db(W.db_codes, W.db_masks)
    s = eng.match(db, eng.prepare(eng.encrypt_query(W.q_codes, W.q_masks, W.eye_ids), 1, "f16_crt"))

    def signed(codes, masks):      # +1 / -1 where the mask is set, else 0: sums below 2^24 are exact in fp32
        c, m = (torch.as_tensor(np.asarray(x)).cuda().float() for x in (codes, masks))
        return m - 2 * c * m

    rc, rm = O.rotated_templates(W.q_codes, W.q_masks, eng.rho)
    want = signed(rc, rm) @ signed(O.unpack(W.db_codes), O.unpack(W.db_masks)).T
    assert torch.equal(eng.decrypt(s).cpu(), want.round().long().cpu())


# rings of which two columns in one block are shorter than its 512 threads (n_eyes * 31 * Lq >= 304), one and two query
# primes, an odd column count among them: by additions (h = 16) and by transforms
@pytest.mark.parametrize("log_n_q,h,L,Lq,n_eyes", [(5, 16, 2, 1, 12), (5, 16, 4, 2, 6), (7, 16, 2, 1, 11), (7, 128, 2, 1, 11),
                                                   (7, 128, 4, 2, 12), (8, 16, 4, 2, 5), (8, 64, 2, 1, 12), (8, 128, 4, 2, 5),
                                                   (9, 16, 4, 2, 12), (9, 64, 4, 2, 12), (10, 16, 2, 1, 12), (13, 16, 2, 1, 1)])
def test_query_encryption_short_columns(log_n_q, h, L, Lq, n_eyes):
    B.build()
    prm = dict(log_n_db=7, log_n_q=log_n_q, n_limbs=L, n_limbs_q=Lq, prime_bits=60, log2_delta=60 if Lq == 2 else 40,
               seed=9)
    P = O.Params(**prm, h=h)
    W = synth.make_workload(n_eyes=n_eyes, n_db=1, seed=21)
    eng = E.Engine(**prm, hamming_weight=h).keygen()
    ct = O.query_encrypt(P, W.q_codes, W.q_masks, W.eye_ids)
    for _ in range(3):
        assert np.array_equal(_u64(eng.encrypt_query(W.q_codes, W.q_masks, W.eye_ids), ct.shape), ct)


def test_graphs_outlive_a_second_keygen():
    """Decryption and normalisation captured before icm_keygen is called again replay on the transform tables that
    they were captured with."""
    B.build()
    prm = dict(log_n_db=9, log_n_q=9, n_limbs=4, n_limbs_q=2, prime_bits=60, log2_delta=60, seed=9)
    W = synth.make_workload(n_eyes=1, n_db=300, seed=21)
    eng = E.Engine(**prm, hamming_weight=16).keygen()
    db, sdb = eng.encrypt_db(W.db_codes, W.db_masks), eng.encrypt_db_slots(W.db_codes, W.db_masks)
    q = eng.prepare(eng.encrypt_query(W.q_codes, W.q_masks, W.eye_ids), 1, "u64")
    s, r = eng.match(db, q), eng.rescale(eng.match(sdb, q))
    qm, dm = torch.as_tensor(W.q_masks).cuda(), torch.as_tensor(W.db_masks).cuda()
    nbytes, wbytes = E.C.icm_normalize_bytes(r.handle)
    ws = torch.empty(wbytes, dtype=torch.uint8, device="cuda")
    want = eng.decrypt(s), eng.normalize(r, qm, dm, ws=ws)
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        got = eng.decrypt(s), eng.normalize(r, qm, dm, ws=ws)
    eng.keygen()
    E.Engine(**{**prm, "seed": 10}, hamming_weight=16).keygen()      # takes what the call above may have given back
    for t in got:
        t.zero_()
    g.replay()
    torch.cuda.synchronize()
    for a, b in zip(got, want):
        assert b.any() and torch.equal(a, b)


def test_decryption_from_two_threads():
    """Two contexts of different rings decrypt from two host threads: no launch meets the other one's limit of
    dynamic shared memory."""
    B.build()
    work = []
    for log_n_db in (5, 12):
        eng = E.Engine(log_n_db=log_n_db, log_n_q=9, n_limbs=2, n_limbs_q=1, prime_bits=60, log2_delta=40, seed=9,
                       hamming_weight=16).keygen()
        W = synth.make_workload(n_eyes=1, n_db=20, seed=21)
        s = eng.match(eng.encrypt_db(W.db_codes, W.db_masks),
                      eng.prepare(eng.encrypt_query(W.q_codes, W.q_masks, W.eye_ids), 1, "u64"))
        out = torch.zeros(31 * 20, dtype=torch.int64, device="cuda")
        work.append((eng, s, out, eng.decrypt(s).flatten(), torch.cuda.Stream()))
    torch.cuda.synchronize()
    errors = []

    def loop(eng, s, out, want, st):
        try:
            for _ in range(4000):
                E.C.icm_decrypt_scores(eng.ctx, s.handle, out, out.numel(), stream=st)
        except Exception as e:
            errors.append(e)

    threads = [threading.Thread(target=loop, args=w) for w in work]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    assert not errors
    for _, _, out, want, _ in work:
        assert torch.equal(out, want)


# chunks whose b-rows go through the transforms (h additions per row would cost more): four columns per block in
# rings of 2^7 to 2^12, two in 2^13; several blocks, partial ones
@pytest.mark.parametrize("log_n_db,h,n_db", [(7, 128, 300), (9, 512, 40), (10, 256, 1100), (11, 512, 90), (12, 512, 100),
                                             (13, 2048, 40)])
def test_database_encryption_by_transforms(log_n_db, h, n_db):
    B.build()
    prm = dict(log_n_db=log_n_db, log_n_q=max(7, (h - 1).bit_length()), n_limbs=2, n_limbs_q=1, prime_bits=60,
               log2_delta=40, seed=9)
    P = O.Params(**prm, h=h)
    W = synth.make_workload(n_eyes=1, n_db=n_db, seed=21)
    eng = E.Engine(**prm, hamming_weight=h).keygen()
    A = O.db_rows(P, W.db_codes, W.db_masks, O.db_layout(n_db, P.ndb, P.rho))
    db = eng.encrypt_db(W.db_codes, W.db_masks)
    assert np.array_equal(_from_digit_form(_u64(db.buf, A.shape), P.q), A)


def _best_ms(f):
    t = []
    for _ in range(4):
        a, b = torch.cuda.Event(True), torch.cuda.Event(True)
        a.record()
        f()
        b.record()
        torch.cuda.synchronize()
        t.append(a.elapsed_time(b))
    return min(t)


def test_few_templates_in_a_large_ring():
    """100 templates store 130 rows of a ring of 2^14: they add about as much again to the time of the a-part's 2^14
    rows, where a transform over the ring and back would add three times as much."""
    B.build()
    eng = E.Engine(log_n_db=14, log_n_q=9, n_limbs=2, n_limbs_q=1, prime_bits=60, log2_delta=40, seed=9).keygen()
    W = synth.make_workload(n_eyes=1, n_db=100, seed=21)
    empty = _best_ms(lambda: eng.encrypt_db(W.db_codes[:0], W.db_masks[:0]))
    assert _best_ms(lambda: eng.encrypt_db(W.db_codes, W.db_masks)) < 3 * empty


def test_messages_of_short_query_rings():
    """The database messages of a query ring of 2^9, too short for words of four entries, cost less than 1.8 times
    those of 2^10 in all of an encryption (2.2 times with words of four)."""
    B.build()
    W = synth.make_workload(n_eyes=1, n_db=2000, seed=21)
    t = []
    for log_n_q in (9, 10):
        eng = E.Engine(log_n_db=12, log_n_q=log_n_q, n_limbs=2, n_limbs_q=1, prime_bits=60, log2_delta=40, seed=9).keygen()
        t.append(_best_ms(lambda: eng.encrypt_db(W.db_codes, W.db_masks)))
    assert t[0] < 1.8 * t[1]


def test_short_query_rings_cost_what_long_ones_do():
    """With few non-zeros in the secrets the additions of a query encryption do not depend on the ring; transforms
    over rings of 2^6 would take six times those over 2^13."""
    B.build()
    W = synth.make_workload(n_eyes=12, n_db=1, seed=21)
    t = []
    for log_n_q in (6, 13):
        eng = E.Engine(log_n_db=6, log_n_q=log_n_q, n_limbs=2, n_limbs_q=1, prime_bits=60, log2_delta=40, seed=9,
                       hamming_weight=16).keygen()
        t.append(_best_ms(lambda: eng.encrypt_query(W.q_codes, W.q_masks, W.eye_ids)))
    assert t[0] < 2.5 * t[1]


@pytest.mark.parametrize("log_n_db,h,n_db,n_eyes", [(7, 128, 300, 1), (8, 256, 700, 2), (9, 512, 40, 1), (10, 512, 2100, 3),
                                                    (12, 512, 4100, 1), (12, 16, 4100, 2), (13, 64, 100, 2)])
def test_decryption_routes(log_n_db, h, n_db, n_eyes):
    """Small rings by transforms (many non-zeros in the secrets) and large ones by additions (few), one and several
    blocks: the cleartext inner products at both levels, with the same error bound."""
    B.build()
    eng = E.Engine(log_n_db=log_n_db, log_n_q=9 if h > 256 else 8, n_limbs=2, n_limbs_q=1, prime_bits=60, log2_delta=40,
                   seed=9, hamming_weight=h).keygen()
    W = synth.make_workload(n_eyes=n_eyes, n_db=n_db, seed=21)
    db = eng.encrypt_db(W.db_codes, W.db_masks)
    s = eng.match(db, eng.prepare(eng.encrypt_query(W.q_codes, W.q_masks, W.eye_ids), n_eyes, "f16_crt"))

    def signed(codes, masks):      # +1 / -1 where the mask is set, else 0: sums below 2^24 are exact in fp32
        c, m = (torch.as_tensor(np.asarray(x)).cuda().float() for x in (codes, masks))
        return m - 2 * c * m

    rc, rm = O.rotated_templates(W.q_codes, W.q_masks, eng.rho)
    want = (signed(rc, rm) @ signed(O.unpack(W.db_codes), O.unpack(W.db_masks)).T).round().long()
    for scores in (s, eng.rescale(s)):
        got, err = eng.decrypt(scores, with_error=True)
        assert torch.equal(got, want) and 0 <= float(err) < 0.25


def test_decryption_of_few_rows_in_a_large_ring():
    """With few non-zeros in the secrets a decryption costs its rows, not its ring (4.2 times as much from N_db = 2^12
    to 2^14 by transforms)."""
    B.build()
    W = synth.make_workload(n_eyes=8, n_db=100, seed=21)
    t = []
    for log_n_db in (12, 14):
        eng = E.Engine(log_n_db=log_n_db, log_n_q=9, n_limbs=4, n_limbs_q=2, prime_bits=60, log2_delta=60, seed=9,
                       hamming_weight=64).keygen()
        s = eng.match(eng.encrypt_db(W.db_codes, W.db_masks),
                      eng.prepare(eng.encrypt_query(W.q_codes, W.q_masks, W.eye_ids), 8, "f16_crt"))
        t.append(_best_ms(lambda: eng.decrypt(s)))
        s = None
    assert t[1] < 2.5 * t[0]


def _normalised(log_n_db, n_db, n_eyes):
    eng = E.Engine(log_n_db=log_n_db, log_n_q=9, n_limbs=4, n_limbs_q=2, prime_bits=60, log2_delta=60, seed=9,
                   hamming_weight=16).keygen()
    W = synth.make_workload(n_eyes=n_eyes, n_db=n_db, seed=21)
    db = eng.encrypt_db_slots(W.db_codes, W.db_masks)
    ct = eng.encrypt_query(W.q_codes, W.q_masks, W.eye_ids)
    r = eng.rescale(eng.match(db, eng.prepare(ct, n_eyes, "f16_crt")))
    return eng, W, r, torch.as_tensor(W.q_masks).cuda(), torch.as_tensor(W.db_masks).cuda()


@pytest.mark.parametrize("log_n_db", [5, 7, 9, 10])
def test_normalisation_of_small_rings(log_n_db):
    """Blocks of 128 threads (rings up to 2^9) and of 512: decoded distances of all the blocks, a partial last
    one among them."""
    B.build()
    eng, W, r, qm, dm = _normalised(log_n_db, 777, 2)
    hd = eng.decrypt_slots(r, eng.normalize(r, qm, dm)).cpu().numpy()
    rc, rm = O.rotated_templates(W.q_codes, W.q_masks, eng.rho)
    ref = O.fractional_hd(*O.hd_counts(rc, rm, O.unpack(W.db_codes), O.unpack(W.db_masks)))
    assert hd.shape == ref.shape and np.abs(hd - ref).max() < 1e-4


def test_normalisation_time_of_small_rings():
    """The same scores in rings of 2^7 and 2^9 take about the same time (1.9 times with blocks of 512 threads)."""
    B.build()
    t = []
    for log_n_db in (7, 9):
        eng, _, r, qm, dm = _normalised(log_n_db, 500, 32)
        out = eng.normalize(r, qm, dm)
        t.append(_best_ms(lambda: eng.normalize(r, qm, dm, out=out)))
    assert t[0] < 1.7 * t[1]
