"""hann_encode_candidates against the oracle's encoding, exactly, over the rings and plaintext counts at which its kernels change: pass A of
four to eight stages, fewer plaintexts than columns of a CTA, rows small enough to skip the reduction of their coefficients and rows that
are not, ragged blocks and padded dimensions, baby-step counts that are and are not multiples of eight."""
import numpy as np
import pytest

from oracle.oracle import find_primes
from paper_2608_21131_b200 import synth
from tests.helpers import make_oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("logN,R,B,bits,norm,dim,short", [
    (12, 8, 8, (50, 50), 1.0, 8, 0),           # four stages: full transforms of the slots
    (13, 8, 8, (50, 40), 1.0, 8, 1),           # five; eight plaintexts, sixty-four columns a CTA
    (13, 16, 8, (30, 30, 30), 1.0, 11, 700),   # coefficients above half the 30-bit primes
    (14, 16, 16, (50,), 1.0, 16, 4000),
    (14, 16, 8, (50, 50), 600.0, 13, 5),       # some coefficients of 2^49 and more, others below
    (15, 8, 8, (50, 45), 1.0, 8, 16000),
    (16, 8, 8, (50, 50), 1.0, 7, 3),
    (16, 8, 8, (50,), 3000.0, 8, 0),
    (14, 16, 4, (50,), 1.0, 12, 9),            # baby steps not a multiple of eight
])
def test_encoded_candidates_equal_the_oracle(logN, R, B, bits, norm, dim, short):
    import torch

    from paper_2608_21131_b200 import binding as b

    q = []
    for w in bits:
        q.append(next(x for x in find_primes(w, logN + 1, len(bits)) if x not in q))
    ps = synth.ParamSet("enc", logN, tuple(q), next(x for x in find_primes(60, logN + 1, 8) if x not in q), 40, R, B, 0)
    c, o = b.Context(ps), make_oracle(ps)
    rng = np.random.default_rng(logN * 7 + R)
    rows = (norm * synth.normalise(rng.standard_normal((ps.n - short, dim)))).astype(np.float32)
    full = np.zeros((ps.n, R), dtype=np.float32)
    full[: rows.shape[0], :dim] = rows
    want = o.encode_block(full).reshape(R, ps.L, ps.N)
    pt = c.encode_candidates(torch.from_numpy(rows).to(c.device), c.workspace(1))
    assert np.array_equal(c.export(b.KIND_PT, pt, R).reshape(R, ps.L, ps.N), want)


@pytest.mark.parametrize("logN,R,B,nb", [(13, 16, 8, 2), (13, 32, 16, 5), (14, 16, 8, 3)])
def test_blocks_on_two_streams_encode_to_the_same_words(logN, R, B, nb):
    """A level of several blocks alternates between two streams and the two halves of the FFT buffer; one block at a time does not."""
    import torch

    from paper_2608_21131_b200 import binding as b

    ps = synth.ParamSet("two", logN, tuple(find_primes(50, logN + 1, 2)), find_primes(60, logN + 1, 1)[0], 40, R, B, 0)
    c = b.Context(ps)
    rows = torch.from_numpy(synth.toy_corpus(5, rows=nb * ps.n - 7, dim=R)).to(c.device)
    ws = c.workspace(nb)
    pt = c.encode_candidates(rows, ws)
    one = torch.cat([c.encode_candidates(rows[i * ps.n:(i + 1) * ps.n].contiguous(), ws) for i in range(nb)])
    torch.cuda.synchronize()
    assert torch.equal(pt, one)


@pytest.mark.parametrize("logN,R,B,nb,two", [
    (13, 16, 8, 2, True), (14, 16, 8, 3, True),
    (13, 16, 8, 1, False),  # one block
    (13, 16, 4, 2, False),  # no half-size FFT: baby steps not a multiple of eight
    (12, 16, 8, 2, False),  # no half-size FFT: four stages in pass A
])
def test_which_levels_encode_on_two_streams(logN, R, B, nb, two):
    """the half-size FFT of one block fills half of the FFT buffer; the second half is written by the blocks of the second stream"""
    import torch

    from paper_2608_21131_b200 import binding as b

    ps = synth.ParamSet("two", logN, tuple(find_primes(50, logN + 1, 2)), find_primes(60, logN + 1, 1)[0], 40, R, B, 0)
    c = b.Context(ps)
    rows = torch.from_numpy(synth.toy_corpus(5, rows=nb * ps.n, dim=R)).to(c.device)
    ws = c.workspace(nb)
    ws.fill_(-1)
    c.encode_candidates(rows, ws)
    torch.cuda.synchronize()
    fft = R * ps.n * 2  # words: one complex number per slot and plaintext
    first, second = ws[: fft // 2], ws[fft // 2 : fft]
    assert bool((first != -1).all())
    half_size = B % 8 == 0 and logN >= 13
    assert bool((second != -1).all()) == (two or not half_size)
    assert bool((second == -1).all()) == (half_size and not two)
    # one lane: the profile of the launches puts all blocks on the context's stream
    if two:
        ws.fill_(-1)
        c.kernel_profile(True)
        c.encode_candidates(rows, ws)
        c.sync()
        c.kernel_profile(False)
        assert bool((second == -1).all())


def test_two_streams_inside_a_graph():
    """the fork to the second stream and the join are captured with the call; a replay on new rows gives the plain call's words"""
    import torch

    from paper_2608_21131_b200 import binding as b

    logN, R, B, nb = 13, 16, 8, 3
    ps = synth.ParamSet("two", logN, tuple(find_primes(50, logN + 1, 2)), find_primes(60, logN + 1, 1)[0], 40, R, B, 0)
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        c = b.Context(ps, stream=stream)
        ws = c.workspace(nb)
        rows = torch.from_numpy(synth.toy_corpus(1, rows=nb * ps.n - 5, dim=R)).to(c.device)
        pt = c.encode_candidates(rows, ws)  # loads every kernel
        c.sync()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream):
            c.encode_candidates(rows, ws, pt)
        for seed in (2, 3):
            rows.copy_(torch.from_numpy(synth.toy_corpus(seed, rows=nb * ps.n - 5, dim=R)))
            want = c.encode_candidates(rows, ws).clone()
            pt.zero_()
            ws.fill_(-1)
            graph.replay()
            c.sync()
            assert torch.equal(pt, want)
            assert bool((ws[R * ps.n : 2 * R * ps.n] != -1).all())  # through both halves of the FFT buffer
    torch.cuda.synchronize()
