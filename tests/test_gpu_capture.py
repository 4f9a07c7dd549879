"""Server-side calls captured into a CUDA graph: the chains are launched with programmatic dependencies and fork to the context's helper
streams, and a replay on new contents of the same buffers must give the bits of the plain call."""
import numpy as np
import pytest

from paper_2608_21131_b200 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("logN,R,B,L,lazy,n_rows", [(10, 16, 4, 2, False, 9000), (12, 32, 8, 3, True, 4200)])
def test_a_captured_level_replays_on_new_inputs(logN, R, B, L, lazy, n_rows):
    import torch

    from paper_2608_21131_b200 import binding as b

    ps = synth.small_params(logN, R, B, L=L, big=L > 2)
    if L > 2:
        ps = ps.with_(log_scale=40)
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        g = b.Context(ps, stream=stream)
        g.set_tuning(b.TUNE_GIANT_LAZY, int(lazy))
        rots = sorted(set(range(1, B + 1)) | {k * B for k in range(1, ps.G)})
        s, evk = g.keygen_seeded(5, rots)
        g.load_keys(evk, rots)
        nb = g.n_blocks(n_rows)
        ws, baby = g.workspace(nb), g.alloc(g.sizeof(b.SIZE_BABY))
        pt, inner = g.alloc(nb * g.sizeof(b.SIZE_PT_BLOCK)), g.alloc(nb * g.sizeof(b.SIZE_INNER))
        score = g.alloc(nb * g.sizeof(b.SIZE_CT))

        def inputs(seed):
            km = synth.key_material(ps, seed, rots=[])
            ct = g.import_(b.KIND_CT, g.encrypt_query(s, synth.toy_query(seed, dim=R), km.ct_a, km.ct_e), 1)
            return ct, torch.from_numpy(synth.toy_corpus(seed, rows=n_rows, dim=R)).to(g.device)

        ct, rows = inputs(1)
        level = lambda: g.query_level(ct, rows, ws, baby, pt, inner, score)
        level()  # loads every kernel
        g.sync()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream):
            level()
        for seed in (1, 2):
            ct_new, rows_new = inputs(seed)
            ct.copy_(ct_new)
            rows.copy_(rows_new)
            level()
            g.sync()
            want = score.clone()
            score.zero_()
            graph.replay()
            g.sync()
            assert torch.equal(score, want) and int(score.abs().max()) > 0
        # and the bits that decrypt: the last inputs' scores
        got = g.decrypt_scores(s, g.export(b.KIND_CT, score, nb)).reshape(-1)[:n_rows]
        exact = synth.toy_corpus(2, rows=n_rows, dim=R).astype(np.float64) @ synth.toy_query(2, dim=R).astype(np.float64)
        assert np.abs(got - exact).max() < 2.0 ** ps.tol_log2
    torch.cuda.synchronize()
