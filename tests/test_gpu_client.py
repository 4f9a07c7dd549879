"""The client's calls over the ways their host buffers can go: pageable ciphertexts below and above the 16 MiB from which a helper thread
shares the upload out, pieces of fewer and more than eight ciphertexts, page-locked buffers, a mix of both, lengths that leave a remainder
of a slot, and two contexts on two threads.  The way of a copy never shows in the bits."""
import threading

import numpy as np
import pytest

from oracle.oracle import find_primes
from paper_2608_21131_b200 import synth
from tests.helpers import make_oracle

pytestmark = pytest.mark.gpu


def context(logN, L, seed=1):
    from paper_2608_21131_b200 import binding as b

    ps = synth.ParamSet("client", logN, tuple(find_primes(45, logN + 1, L)), find_primes(60, logN + 1, 1)[0], 30, 8, 4, 0)
    return b.Context(ps), ps, synth.key_material(ps, seed, rots=[])


def pinned(a):
    import torch

    t = torch.empty(a.shape, dtype=torch.int64 if a.dtype == np.uint64 else torch.from_numpy(a).dtype).pin_memory().numpy().view(a.dtype)
    t[...] = a
    return t


def decrypted(c, s, ct, scores):
    """the library's call on these very buffers (real parts)"""
    c._ck(c.lib.hann_decrypt_scores(c.h, s.ctypes.data, ct.ctypes.data, ct.shape[0], 60, scores.ctypes.data, None))
    return scores


# MiB of a piece: 1, 15 and 16; 17 ciphertexts are two pieces of 16 and one of 2 (the slots are used again); polynomials of 2.75 MiB
# are five slots and a half; ciphertexts of 15 MiB go through in pieces of fewer than eight
@pytest.mark.parametrize("logN,L,count", [(13, 1, 9), (16, 3, 5), (15, 4, 8), (15, 4, 17), (15, 11, 3), (16, 15, 5)])
def test_decryption_of_pageable_and_page_locked_buffers(logN, L, count):
    c, ps, km = context(logN, L)
    rng = np.random.default_rng(logN + L)
    ct = rng.integers(0, min(ps.q), size=(count, 2, L, ps.N), dtype=np.uint64)
    alone = np.stack([c.decrypt_scores(km.s, ct[i:i + 1], log_scale_out=60)[0] for i in range(count)])
    for cts in (ct, pinned(ct)):
        for scores in (np.full((count, ps.n), np.nan), pinned(np.full((count, ps.n), np.nan))):
            assert np.array_equal(decrypted(c, km.s, cts, scores), alone)
    got, imag = c.decrypt_scores(km.s, ct, log_scale_out=60, want_imag=True)
    assert np.array_equal(got, alone) and np.isfinite(imag).all() and np.abs(imag).max() > 0
    ct[...] = 0  # the call has read its buffers when it returns
    assert not np.array_equal(c.decrypt_scores(km.s, ct, log_scale_out=60), alone)


@pytest.mark.parametrize("logN,L", [(10, 2), (14, 4), (16, 3)])
def test_encryption_of_pageable_and_page_locked_buffers(logN, L):
    c, ps, km = context(logN, L)
    q = synth.toy_query(3, dim=5)
    want = make_oracle(ps).encrypt_query(km.s, q, km.ct_a, km.ct_e)
    for a in (km.ct_a, pinned(km.ct_a)):
        for out in (np.zeros_like(want), pinned(np.zeros_like(want))):
            c._ck(c.lib.hann_encrypt_query(c.h, km.s.ctypes.data, q.ctypes.data, 5, a.ctypes.data, km.ct_e.ctypes.data, out.ctypes.data))
            assert np.array_equal(out, want)
    # the uniform half is where the ciphertext wants it already
    out = np.zeros_like(want)
    out[1] = km.ct_a
    c._ck(c.lib.hann_encrypt_query(c.h, km.s.ctypes.data, q.ctypes.data, 5, out[1].ctypes.data, km.ct_e.ctypes.data, out.ctypes.data))
    assert np.array_equal(out, want)


def test_two_contexts_decrypt_on_two_threads():
    jobs = []
    for seed in (1, 2):
        c, ps, km = context(15, 4, seed)
        ct = np.random.default_rng(seed).integers(0, min(ps.q), size=(10, 2, 4, ps.N), dtype=np.uint64)
        jobs.append((c, km.s, ct, np.stack([c.decrypt_scores(km.s, ct[i:i + 1], log_scale_out=60)[0] for i in range(10)]), []))

    def work(c, s, ct, want, bad):
        for _ in range(20):
            if not np.array_equal(c.decrypt_scores(s, ct, log_scale_out=60), want):
                bad.append(1)

    threads = [threading.Thread(target=work, args=j) for j in jobs]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not any(j[4] for j in jobs)
