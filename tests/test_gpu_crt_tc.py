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
    W = synth.make_workload(n_eyes=26, n_db=231, seed=31)
    cuts = [0, 1, 150, 231]
    dbs = [eng.encrypt_db(W.db_codes[a:b], W.db_masks[a:b], chunk_id=i) for i, (a, b) in enumerate(zip(cuts, cuts[1:]))]
    return eng, W, dbs


@pytest.mark.parametrize("n_eyes", [1, 8, 9, 16, 17, 24, 25])
def test_column_groups(setup, n_eyes):
    eng, W, dbs = setup
    ct = eng.encrypt_query(W.q_codes[:n_eyes], W.q_masks[:n_eyes], W.eye_ids[:n_eyes])
    q = eng.prepare(ct, n_eyes, "f16_crt")
    res = {}
    try:
        for v in (256, 1, 2, 3):
            C.icm_ctx_set_variant(eng.ctx, v)
            outs = eng.match_batch(dbs, q)
            torch.cuda.synchronize()
            res[v] = [s.residues() for s in outs]
    finally:
        C.icm_ctx_set_variant(eng.ctx, 0)
    C.icm_device_status(True)
    for v in (1, 2, 3):
        for a, b in zip(res[v], res[256]):
            assert np.array_equal(a, b), v


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
