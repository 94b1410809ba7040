"""Mask sampler at the edges of its steps: rows around one word and around a warp's 512 keys, odd and
even seed counts, one seed and more, windows and anchors at their extremes."""
import numpy as np
import pytest
import torch

from paper_2607_21927_gb300 import ris
from test_gpu_mask import check_rows, gpu_mask, oracle_spec

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N", [2, 31, 64, 511, 514, 2050])
@pytest.mark.parametrize("S", [1, 2, 3, 5])
@pytest.mark.parametrize("mode,W,A,head_keyed,sampler", [
    (0, 1, 0, False, 0), (1, 1, 5, True, 0), (0, 2**31 - 1, 0, False, 0), (0, 1, 2**31 - 1, False, 0),
    (1, 700, 33, False, ris.SAMPLER_DRAWS)])
def test_mask_steps(N, S, mode, W, A, head_keyed, sampler):
    seeds = [11 + 7 * s for s in range(S)]
    m = gpu_mask(N, mode, 0.07, seeds, kv_heads=2, W=W, A=A, per_head=head_keyed, layer_key=3, sampler=sampler)
    heads = range(2) if head_keyed else [0]
    specs = [oracle_spec(N, mode, 0.07, seeds, W=min(W, N), A=min(A, N), head_key=h, layer_key=3, sampler=sampler)
             for h in heads]
    rows = np.unique(np.clip([0, 1, 30, 31, 32, 510, 511, 512, 513, 2047, 2048, 2049, N - 2, N - 1], 0, N - 1))
    check_rows(m, specs, rows)


@pytest.mark.parametrize("N,heads,mode,W,A", [
    (2430, 4, 0, 1, 0),     # 9720 rows: one below the line of four rows per block
    (2433, 4, 0, 1, 0),     # 9732: just above it
    (2050, 5, 1, 700, 33),  # 10250: the last block has two rows
    (9729, 1, 0, 1, 0)])
def test_one_seed_rows(N, heads, mode, W, A):
    m = gpu_mask(N, mode, 0.03, [77], kv_heads=heads, W=W, A=A, per_head=heads > 1, layer_key=5)
    specs = [oracle_spec(N, mode, 0.03, [77], W=W, A=A, head_key=h, layer_key=5) for h in range(heads)]
    check_rows(m, specs, np.unique([0, 1, 2, 3, 4, 31, 511, 512, 513, 2047, 2048, N - 3, N - 2, N - 1]))


@pytest.mark.parametrize("N,mode,d,S,W,A", [
    (1500, 0, 0.5, 256, 1, 0), (1500, 0, 0.3, 71, 1, 40), (2050, 1, 0.4, 30, 90, 0),  # full steps, some of them at the last seed
    (1100, 0, 0.25, 23, 1, 700), (1100, 0, 0.02, 6, 1, 1024), (900, 0, 0.999, 3, 1, 0), (1500, 0, 0.1, 70, 1, 0)])
def test_steps_that_fill_up(N, mode, d, S, W, A):
    seeds = [5 + 3 * s for s in range(S)]
    m = gpu_mask(N, mode, d, seeds, W=W, A=A, layer_key=2)
    rows = np.unique(np.clip([0, 1, 31, 32, 511, 512, 513, 700, 1023, 1024, 1025, N - 2, N - 1], 0, N - 1))
    check_rows(m, [oracle_spec(N, mode, d, seeds, W=W, A=A, layer_key=2)], rows)


def test_kept_keys_cost_no_more_draws():
    """Once every key is kept, by the seeds before or as an anchor, further seeds cost next to nothing."""
    def us(d, S, A):
        best = float("inf")
        for _ in range(4):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            gpu_mask(8192, 0, d, list(range(S)), A=A).free()
            b.record()
            b.synchronize()
            best = min(best, a.elapsed_time(b) * 1e3)
        return best
    t = {k: us(*k) for k in ((0.5, 32, 0), (0.5, 256, 0), (0.3, 70, 0), (0.1, 256, 0), (0.1, 70, 0), (0.01, 70, 0), (0.01, 70, 8192))}
    print({k: round(v) for k, v in t.items()})
    assert t[0.5, 256, 0] <= 1.5 * t[0.5, 32, 0]
    assert t[0.01, 70, 8192] <= 0.5 * t[0.01, 70, 0]
