"""The key-switch kernels (lift, digit product with the sum over rotations, final combination) on residues drawn directly, at the
edges of their dispatch: one to nine digits, one to five blocks, moduli of every arithmetic class side by side, neighbouring moduli
of very different size, residues at the ends of their range, and buffers that are only 8-byte aligned.  Exact against the oracle."""
import numpy as np
import pytest

from oracle.oracle import find_primes
from paper_2608_21131_b200 import synth
from tests.helpers import make_oracle

pytestmark = pytest.mark.gpu


def edge_residues(seed, q, N, lead):
    a = synth.uniform_residues(seed, 1, list(q), N, lead=lead)
    for i, m in enumerate(q):
        a[..., i, 0:6] = (0, 1, m - 1, m // 2, m // 2 + 1, m // 2 - 1)
        a[0, ..., i, :] = m - 1 if lead[0] > 1 else a[0, ..., i, :]
    return a


@pytest.mark.parametrize(
    "logN,bits,pbits,nb",
    [
        (10, (50,), 60, 3),                     # one digit, whose only modulus is its own
        (10, (30, 30), 31, 5),                  # the special prime below 2^50 as well
        (11, (50, 40, 30), 60, 2),              # source moduli far above the target's: the coefficient is folded first
        (12, (50,) * 4, 60, 4),                 # four items per CTA, one round
        (12, (50,) * 4, 60, 5),                 # and a remainder
        (11, (58, 54, 45, 45, 45), 62, 3),      # every arithmetic class, two items per CTA
        (10, (45,) * 9, 60, 2),                 # more than eight digits: two exact sums per position
        (13, (50,) * 4, 60, 1),
        (15, (50, 50), 60, 2),                  # second lift round of three stages
        (10, (50,) * 3, 62, 5),                 # five and six items go two per CTA, four and seven four
        (10, (50,) * 4, 62, 6),
        (10, (50,) * 4, 62, 7),
        (10, (50,) * 3, 60, 6),                 # (with auxiliary primes)
        (10, (50,) * 3, 60, 4),
    ],
)
def test_rotate_sum_on_edge_residues(logN, bits, pbits, nb):
    import torch

    from paper_2608_21131_b200 import binding as b

    q = []
    for w in bits:
        q.append(next(x for x in find_primes(w, logN + 1, len(bits)) if x not in q))
    p = next(x for x in find_primes(pbits, logN + 1, len(bits) + 1) if x not in q)
    R, B = 16, 4
    ps = synth.ParamSet("edge", logN, tuple(q), p, 20, R, B, 0)
    G, N, L = ps.G, ps.N, ps.L
    rots = [1, 2, 3] + [g * B for g in range(1, G)]
    c, o = b.Context(ps), make_oracle(ps)
    km = synth.key_material(ps, logN, rots=rots)
    evk = {r: o.evk_gen(km.s, r, km.evk_a[i], km.evk_e[i]) for i, r in enumerate(rots)}
    c.load_keys(np.stack([evk[r] for r in rots]), rots)
    inner = edge_residues(7, q, N, (nb * G, 2))
    dev = c.import_(b.KIND_CT, inner, nb * G)
    ws = c.workspace(nb)
    giant = np.stack([evk[g * B] for g in range(1, G)])
    inner = inner.reshape(nb, G, 2, L, N)
    want = np.stack([o.rotate_sum(inner[i], evk[B]) for i in range(nb)])
    want_lazy = np.stack([o.rotate_sum_lazy(inner[i], giant) for i in range(nb)])
    odd = c.alloc(dev.numel() * 8 + 8)[1:]
    odd.copy_(dev)
    for src in (dev, odd):
        assert np.array_equal(c.export(b.KIND_CT, c.rotate_sum(src, nb, ws), nb), want)
        assert np.array_equal(c.export(b.KIND_CT, c.rotate_sum_lazy(src, nb, ws), nb), want_lazy)
    # the hoisted rotations: three keys, one digit set
    baby = c.query_prepare(dev[: 2 * L * N], ws)
    got = c.export(b.KIND_CT, baby, B)
    for r in (1, 2, 3):
        assert np.array_equal(got[r], o.rotate(inner[0, 0], r, evk[r])), r
    torch.cuda.synchronize()


@pytest.mark.parametrize(
    "logN,bits,pbits,nb",
    [
        (10, (50,) * 3, 60, 3),            # three primes: all auxiliary, the lifted polynomials in the place of the digits
        (11, (58, 46, 45, 46), 60, 3),     # a prime of 2^50 and more between them, the digits of which are longer
        (12, (50, 50, 50, 40), 60, 2),     # a ciphertext prime far below the auxiliary ones
        (10, (50,) * 4, 61, 2),            # the largest special prime they stand for
        (10, (50,) * 4, 51, 5),            # and the smallest
        (10, (50, 50, 48), 60, 2),         # the smallest a quarter of the others
        (10, (50, 50, 47), 60, 2),         # primes of too different size, and too few of them: the special prime itself
        (11, (58, 45, 46, 46, 45), 60, 1),  # neighbouring sizes, whichever lies closer to its power of two
        (10, (50, 50, 58), 60, 2),
        (14, (50,) * 4, 60, 1),            # second lift round of two stages
        (14, (45,) * 8, 60, 1),            # the longest chain of that ring, and one that takes the special prime itself
        (14, (45,) * 9, 60, 1),
    ],
)
def test_rotate_sum_through_auxiliary_primes(logN, bits, pbits, nb):
    test_rotate_sum_on_edge_residues(logN, bits, pbits, nb)


@pytest.mark.parametrize("logN,bits", [(10, (50,)), (12, (50, 40)), (11, (50, 58, 45)), (12, (50,) * 4), (13, (50,) * 4), (11, (45,) * 5)])
def test_hoisted_rotations_of_an_unaligned_ciphertext(logN, bits):
    """a ciphertext that is only 8-byte aligned is copied before its inverse transform: the oracle's bits from either"""
    import torch

    from paper_2608_21131_b200 import binding as b

    q = []
    for w in bits:
        q.append(next(x for x in find_primes(w, logN + 1, len(bits)) if x not in q))
    ps = synth.ParamSet("odd", logN, tuple(q), find_primes(60, logN + 1, 1)[0], 20, 16, 4, 0)
    rots = [1, 2, 3]
    c, o = b.Context(ps), make_oracle(ps)
    km = synth.key_material(ps, logN, rots=rots)
    evk = {r: o.evk_gen(km.s, r, km.evk_a[i], km.evk_e[i]) for i, r in enumerate(rots)}
    c.load_keys(np.stack([evk[r] for r in rots]), rots)
    ct = edge_residues(5, q, ps.N, (1, 2))
    dev = c.import_(b.KIND_CT, ct, 1)
    odd = c.alloc(dev.numel() * 8 + 8)[1:]
    odd.copy_(dev)
    ws = c.workspace(1)
    for src in (dev, odd):
        baby = c.export(b.KIND_CT, c.query_prepare(src, ws), 4)
        hoisted = c.export(b.KIND_CT, c.rotate_hoisted(src, 2, 2, ws), 2)
        for r in rots:
            want = o.rotate(ct[0], r, evk[r])
            assert np.array_equal(baby[r], want), r
            assert r == 1 or np.array_equal(hoisted[r - 2], want), r
    torch.cuda.synchronize()


def takes_auxiliary_primes(c, call):
    """whether the ModDown of the call's key switches went through auxiliary primes: it is a launch class of its own"""
    c.kernel_profile(True)
    call()
    c.sync()
    launches = c.kernel_times()["moddown_lift"][1]
    c.kernel_profile(False)
    return launches > 0


@pytest.mark.parametrize(
    "logN,bits,pbits,taken",
    [
        (10, (50,) * 3, 60, True),
        (11, (45,) * 5, 60, True),
        (12, (50, 50, 50, 40), 60, True),      # the three largest are what counts
        (10, (58, 45, 45, 45), 61, True),
        (10, (50,) * 4, 51, True),
        (10, (50,) * 4, 50, False),            # a special prime that the FP64 pipe transforms itself
        (10, (50,) * 4, 62, False),            # and one above what the recombination holds
        (10, (50, 50), 60, False),
        (10, (50, 50, 58), 60, False),         # too few primes below 2^50
        (10, (50, 50, 48), 60, True),          # a quarter of the others
        (10, (50, 50, 47), 60, False),         # an eighth: too different in size
        (15, (58, 46, 45, 46), 60, True),      # the short chains of the membership circuit
        (14, (45,) * 8, 60, True),             # 2^17 words a polynomial
        (14, (45,) * 9, 60, False),            # and more, on a chain of more than four primes
        (15, (45,) * 5, 60, False),
        (16, (45,) * 4, 60, True),
        (10, (37,) * 9, 60, False),            # the products do not stay below a quarter of three primes
    ],
)
def test_which_chains_take_auxiliary_primes(logN, bits, pbits, taken):
    import torch

    from paper_2608_21131_b200 import binding as b

    q = []
    for w in bits:
        q.append(next(x for x in find_primes(w, logN + 1, len(bits)) if x not in q))
    ps = synth.ParamSet("rule", logN, tuple(q), next(x for x in find_primes(pbits, logN + 1, len(bits) + 1) if x not in q), 20, 16, 4, 0)
    c = b.Context(ps)
    rots = [1, 2, 3, 4, 8, 12]
    c.load_keys(synth.uniform_residues(3, 2, q + [ps.p], ps.N, lead=(len(rots), ps.L, 2)), rots)
    ws = c.workspace(1)
    inner = torch.randint(0, min(q), (c.sizeof(b.SIZE_INNER) // 8,), dtype=torch.int64, device=c.device)
    ct = inner[: 2 * ps.L * ps.N].clone()
    assert takes_auxiliary_primes(c, lambda: c.rotate_sum(inner, 1, ws)) == taken
    assert takes_auxiliary_primes(c, lambda: c.rotate_sum_lazy(inner, 1, ws)) == taken
    assert takes_auxiliary_primes(c, lambda: c.fold(ct, 4, 2, ws)) == taken
    # keys without the words: hoisted rotations, a fold by other strides, one that takes both kinds
    assert not takes_auxiliary_primes(c, lambda: c.query_prepare(ct, ws))
    assert not takes_auxiliary_primes(c, lambda: c.fold(ct, 1, 2, ws))
    assert not takes_auxiliary_primes(c, lambda: c.fold(ct, 2, 2, ws))


@pytest.mark.parametrize("L", [3, 4])
def test_folds_with_and_without_auxiliary_words(L):
    """the keys of multiples of B have words modulo the auxiliary primes, the others have not: folds of either kind, and one that
    takes both, to the oracle's bits"""
    from paper_2608_21131_b200 import binding as b

    logN, R, B = 11, 16, 4
    q = find_primes(50, logN + 1, L)
    ps = synth.ParamSet("fold", logN, tuple(q), find_primes(60, logN + 1, 1)[0], 20, R, B, 0)
    rots = [1, 2, 4, 8]
    c, o = b.Context(ps), make_oracle(ps)
    km = synth.key_material(ps, logN, rots=rots)
    evk = {r: o.evk_gen(km.s, r, km.evk_a[i], km.evk_e[i]) for i, r in enumerate(rots)}
    c.load_keys(np.stack([evk[r] for r in rots]), rots)
    ct = edge_residues(9, q, ps.N, (1, 2))
    for stride, steps in ((1, 2), (4, 2), (1, 4)):
        want = ct[0]
        for t in range(steps):
            rot = o.rotate(want, stride << t, evk[stride << t])
            want = np.stack([(want[:, i] + rot[:, i]) % np.uint64(q[i]) for i in range(L)], axis=1)
        dev = c.fold(c.import_(b.KIND_CT, ct, 1), stride, steps, c.workspace(1))
        assert np.array_equal(c.export(b.KIND_CT, dev, 1)[0], want), (stride, steps)


def test_only_giant_step_keys_take_memory_for_auxiliary_words():
    """loading the keys of the baby steps takes 2 L (L + 1) polynomials each and no more; those of giant steps 6 L more"""
    import torch

    from paper_2608_21131_b200 import binding as b

    logN, L, R, B = 14, 4, 64, 16
    q = find_primes(50, logN + 1, L)
    ps = synth.ParamSet("mem", logN, tuple(q), find_primes(60, logN + 1, 1)[0], 20, R, B, 0)
    c = b.Context(ps)
    keys = synth.uniform_residues(3, 2, q + [ps.p], ps.N, lead=(1, L, 2))

    def taken(rots):
        torch.cuda.synchronize()
        before = torch.cuda.mem_get_info(c.device)[0]
        for r in rots:
            c.load_keys(keys, [r])
        torch.cuda.synchronize()
        return before - torch.cuda.mem_get_info(c.device)[0]

    taken([1])  # the exchange scratch
    key, aux = (2 * L * w * ps.N * 8 for w in (L + 1, 3))
    page = 2 << 20  # what the device allocates in
    assert 14 * key <= taken(range(2, 16)) < 14 * (key + page)
    assert 3 * (key + aux) <= taken([16, 32, 48]) < 3 * (key + aux + 2 * page)


def test_lazy_round_of_many_giant_steps():
    """15 blocks x 511 giant steps in one round: 7,665 polynomials of nine limbs, more than one launch covers (65535 / 9).  A large
    workspace only means larger rounds: the same bits as with rounds of one block"""
    import torch

    from paper_2608_21131_b200 import binding as b

    logN, L, nb = 10, 9, 15
    q = find_primes(45, logN + 1, L)
    ps = synth.ParamSet("many", logN, tuple(q), find_primes(60, logN + 1, 1)[0], 20, 512, 1, 0)
    c = b.Context(ps)
    c.set_tuning(b.TUNE_LAZY_LANES, 1)
    keys = synth.uniform_residues(3, 2, q + [ps.p], ps.N, lead=(5, L, 2))
    for r in range(1, ps.G):
        c.load_keys(keys[r % 5][None], [r])
    inner = torch.randint(0, min(q), (nb * c.sizeof(b.SIZE_INNER) // 8,), dtype=torch.int64, device=c.device,
                          generator=torch.Generator(c.device).manual_seed(4))
    one = c.rotate_sum_lazy(inner, nb, c.workspace(1))
    all_ = c.rotate_sum_lazy(inner, nb, c.alloc((nb + 1) * c.workspace_bytes(1)))
    c.sync()
    assert torch.equal(one, all_)


def test_contexts_of_different_chains_on_two_threads():
    """a call of a five-prime and one of a fifteen-prime context use the same kernel instance with different amounts of shared memory;
    driven by two threads at once, neither takes its limit from the other"""
    import threading

    import torch

    from paper_2608_21131_b200 import binding as b

    logN, calls = 10, 150
    q = find_primes(45, logN + 1, 15)
    p = find_primes(60, logN + 1, 1)[0]

    class Worker(threading.Thread):
        def __init__(self, L):
            super().__init__()
            self.ps = synth.ParamSet("chain", logN, tuple(q[:L]), p, 20, 64, 1, 0)
            self.stream = torch.cuda.Stream()
            self.c = c = b.Context(self.ps, stream=self.stream)
            c.load_keys(synth.uniform_residues(L, 2, q[:L] + [p], self.ps.N, lead=(1, L, 2)), [1])
            self.inner = torch.randint(0, min(q), (c.sizeof(b.SIZE_INNER) // 8,), dtype=torch.int64, device=c.device,
                                       generator=torch.Generator(c.device).manual_seed(L))
            self.ws, self.score = c.workspace(1), c.alloc(c.sizeof(b.SIZE_CT))
            torch.cuda.synchronize()
            self.want = c.rotate_sum(self.inner, 1, self.ws)
            c.sync()
            self.error = None

        def run(self):
            try:
                for _ in range(calls):  # 63 giant steps each
                    self.c.rotate_sum(self.inner, 1, self.ws, self.score)
                self.c.sync()
            except b.HannError as e:
                self.error = e

    workers = [Worker(5), Worker(15)]
    for w in workers:
        w.start()
    for w in workers:
        w.join()
    torch.cuda.synchronize()
    for w in workers:
        assert w.error is None, w.error
        assert torch.equal(w.score, w.want)
