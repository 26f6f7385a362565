"""The decode step's kernel instances at the edges of their ranges: chunks per unit around 256, 512, 1024 and 2048 (beyond that
the general kernel), chunk sizes that are and are not a multiple of a tile or of eight, and steps right after appends."""
import numpy as np
import pytest
import torch

import hkv_inputs as hi

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_chunks,cs", [(1, 32), (255, 8), (256, 32), (257, 16), (512, 8), (513, 24), (1024, 8), (1025, 8),
                                         (2048, 8), (2049, 8), (300, 12)])
def test_chunk_counts_around_the_instances_limits(n_chunks, cs):
    import parity_util as P
    C = n_chunks * cs - (3 if n_chunks > 1 else 0)
    L = hi.tiny(seed=71, B=2, C=C, chunk_size=cs, w=4, Hq=14, Hkv=2, d=128, budget_fraction=0.15, n_steps=2, ragged=C > 200,
                head_type=[[1, 0], [1, 1]])
    P.compare_layer(L)


def test_append_and_decode_interleaved_over_layers():
    """Two layers' appends and steps without any wait between them, against the same calls with a wait after each."""
    from paper_2604_05887_b200.layer import LayerCache, to_device_bf16
    Ls = [hi.cfg1(layer=l, C=2048, block=256, n_steps=1) for l in range(2)]
    q = [to_device_bf16(L.q[0]) for L in Ls]
    g = torch.Generator(device="cuda").manual_seed(7)
    new = [torch.randn(6, 2, 2, 1, 4, 128, device="cuda", generator=g).bfloat16().contiguous()]

    def run(wait):
        lcs = [LayerCache(L, append_capacity=8) for L in Ls]
        outs = []
        for t in range(6):
            for i, lc in enumerate(lcs):
                lc.append(new[0][t, i, 0], new[0][t, i, 1])
                if wait:
                    torch.cuda.synchronize()
                outs.append(lc.new_out())
                lc.decode(q[i], outs[-1])
                if t % 2:
                    outs.append(lc.new_out())
                    lc.decode(q[1 - i], outs[-1])     # a second step of the same cache, not the first after the append
                if wait:
                    torch.cuda.synchronize()
        torch.cuda.synchronize()
        res = [o.view(torch.int16).cpu().numpy() for o in outs]
        for lc in lcs:
            lc.close()
        return res

    want = run(True)
    for _ in range(3):
        assert all(np.array_equal(a, b) for a, b in zip(run(False), want))


def test_a_recorded_step_does_not_stand_for_the_first_after_an_append():
    """A decode call recorded between an append and the next step has not run: the step must still wait for the append (a
    launch that need not may read the cache's tables and rows while the append writes them).  The recording itself
    waits for nothing, so the append may still be on its way when the step is launched."""
    from paper_2604_05887_b200.layer import LayerCache, to_device_bf16
    L = hi.cfg1(layer=0, C=2048, block=256, n_steps=1)
    q = to_device_bf16(L.q[0])
    g = torch.Generator(device="cuda").manual_seed(9)
    new = torch.randn(12, 2, 1, 4, 128, device="cuda", generator=g).bfloat16().contiguous()
    ballast = torch.randn(4096, 4096, device="cuda")

    def run(recorded):
        lc = LayerCache(L, append_capacity=12)
        spare, side, outs, graphs = lc.new_out(), torch.cuda.Stream(), [], []
        lc.decode(q, spare)
        torch.cuda.synchronize()
        for t in range(12):
            if recorded:
                ballast @ ballast                      # keeps the append waiting while the step is recorded
            lc.append(new[t, 0], new[t, 1])
            if recorded:
                with torch.cuda.stream(side):
                    graphs.append(torch.cuda.CUDAGraph())
                    graphs[-1].capture_begin(capture_error_mode="relaxed")
                    lc.decode(q, spare)
                    graphs[-1].capture_end()
            else:
                torch.cuda.synchronize()
            outs.append(lc.new_out())
            lc.decode(q, outs[-1])
        torch.cuda.synchronize()
        res = [o.view(torch.int16).cpu().numpy() for o in outs]
        lc.close()
        return res

    assert all(np.array_equal(a, b) for a, b in zip(run(True), run(False)))
